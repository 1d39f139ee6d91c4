"""The L2 x L2 rows evaluated from their staged columns, where the kernel's
lanes and words can go wrong: few rows, more than 32 electrons, several words
per string, orbitals across word boundaries, and lists in which no two
functions couple (whose columns are not staged)."""
import numpy as np
import pytest

from gpu_util import FP64_FALLBACK, check_elements, l2_csr_cond
from oracle import coracle
from paper_1709_03005_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


def _check(P, couples=True):
    import torch
    from paper_1709_03005_gb300 import hb
    o = coracle.Oracle(P)
    rp, cols, vals = o.l2_csr()
    assert couples == (len(cols) > P.n_l2)
    H = hb.Hamiltonian(P)
    for precision in (hb.HB_FP64, hb.HB_MIXED):
        b = H.allocate()
        b["val"].fill_(float("nan"))
        b["col"].fill_(-1)
        H.build(precision, blocks=b)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(b["row_ptr"].cpu().numpy(), rp)
        np.testing.assert_array_equal(b["col"].cpu().numpy()[: rp[-1]], cols)
        check_elements(b["val"].cpu().numpy()[: rp[-1]], vals, l2_csr_cond(o, rp, cols), 1e-12, FP64_FALLBACK, "L2")
    H.close()


@pytest.mark.parametrize("n_to,n_elec,n_words,n_l2", [(6, 4, 1, 2), (6, 4, 1, 9), (10, 6, 1, 33), (10, 6, 3, 200),
                                                      (10, 6, 4, 65), (34, 40, 1, 150), (40, 66, 4, 70),
                                                      (68, 6, 2, 300)])
def test_values_match_oracle(n_to, n_elec, n_words, n_l2):
    _check(synth.make_problem("l2v", 3, n_to, 2, n_elec, 4, 1, n_l2, 6, n_words=n_words, e_core=0.25))


def test_rows_that_do_not_couple():
    """Two functions four substitutions apart: only the diagonal entries."""
    P = synth.make_problem("l2v", 3, 12, 2, 6, 4, 1, 2, 6)
    P.l2_dets = np.stack([synth.occ_to_words(range(4), range(3), 1), synth.occ_to_words(range(4, 8), range(3, 6), 1)])
    _check(P, couples=False)

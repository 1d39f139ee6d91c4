"""Class 4 on the tensor cores where its tiles and chunks can go wrong: one
orbital, a whole tile, one more than a tile, ranges that start off a multiple
of 8, 1 to 64 states, rows of no term and of several accumulation chunks (256
terms), and fewer slices."""
import numpy as np
import pytest

from gpu_util import MIXED_C4_FALLBACK, MIXED_C4_TC_ABS, check_elements
from oracle import coracle
from paper_1709_03005_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


def _hlc(P, **kw):
    import torch
    from paper_1709_03005_gb300 import hb
    H = hb.Hamiltonian(P, class4_path=2, **kw)
    b = H.allocate()
    b["Hlc"].fill_(float("nan"))
    H.build(hb.HB_MIXED, blocks=b)
    torch.cuda.synchronize()
    assert "class4 tensor cores" in H.tuning_report()
    out = b["Hlc"].cpu().numpy()
    H.close()
    return out


def _case(n_co, cf, cn, n_state, **kw):
    kw = dict(dict(n_to=12, n_elec=6, n_det=80, n_l2=40), **kw)
    return synth.make_tiny(9, n_co=n_co, n_state=n_state, cont_ranges=[(cf, cn)], **kw)


CASES = [(1, 0, 1, 1, {}), (9, 7, 2, 3, {}), (128, 0, 128, 2, {}), (140, 7, 128, 33, {}), (160, 8, 129, 5, {}),
         (270, 5, 264, 2, dict(n_to=30)), (24, 3, 20, 64, dict(n_to=18, n_det=2000, n_l2=30)),
         (24, 1, 9, 2, dict(n_to=34, n_elec=40, n_l2=60))]


@pytest.mark.parametrize("case", CASES, ids=[str(c[:4]) for c in CASES])
def test_tiles(case):
    P = _case(*case[:4], **case[4])
    o = coracle.Oracle(P)
    check_elements(_hlc(P), o.class4_rows(0, P.n_l2), o.class4_rows_abs(0, P.n_l2), 1e-10, MIXED_C4_FALLBACK, "class 4",
                   abs_frac=MIXED_C4_TC_ABS)


@pytest.mark.parametrize("slices", [3, 4, 5])
def test_slices(slices):
    """S digits of 8 bits a factor, products of S(S + 1) / 2 pairs: a term is off by at
    most (S + 3) 2^(-8 S) of the largest integral times the largest coefficient, taken up to a power of two each."""
    P = _case(140, 7, 128, 33)
    o = coracle.Oracle(P)
    x = max(np.abs(P.eri_tttc).max(), np.abs(P.h).max())
    c = max(np.abs(g.ci).max() for g in P.groups)
    pairs = np.bitwise_count(P.l2_dets.reshape(P.n_l2, 1, -1) ^ P.groups[0].dets.reshape(1, P.groups[0].dets.shape[0], -1)).sum(-1)
    terms = (2 * (pairs == 3) + 13 * (pairs == 1)).sum(1, keepdims=True)
    d = np.abs(_hlc(P, split_slices=slices) - o.class4_rows(0, P.n_l2))
    assert (d <= 4 * (slices + 3) * 2.0 ** (-8 * slices) * x * c * terms).all(), d.max()

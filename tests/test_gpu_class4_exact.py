"""Class 4 on the tensor cores with sums as large as they get: what is to be exact is."""
import numpy as np
import pytest

from oracle import coracle
from paper_1709_03005_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


def _coherent_terms():
    """One L2 function with 304 partners that give one integral each (holes of both
    spins, a beta particle).  Integrals and coefficients have three base-256 digits,
    255, about 127, about 127, and the signs of the coefficients make every term
    positive: the sums of each accumulator are the largest there are."""
    n_to, n_co, na, nb = 24, 9, 4, 4                       # electrons of the L2 function
    P = synth.make_tiny(3, n_to=n_to, n_co=n_co, n_elec=na + nb - 1, n_det=1, n_state=1, n_l2=1)
    a, b = (1 << na) - 1, (1 << nb) - 1
    dets = [(a & ~(1 << h1), (b & ~(1 << h2)) | 1 << q) for h1 in range(na) for h2 in range(nb) for q in range(nb, nb + 19)]
    P.l2_dets = np.array([[a, b]], dtype=np.uint64)
    P.groups[0].dets = np.array(dets, dtype=np.uint64)
    dx = np.array([255, 127, 127])
    rng = np.random.default_rng(0)
    dc = np.stack([np.full(len(dets), 255), rng.integers(120, 128, len(dets)), rng.integers(120, 128, len(dets))], 1)
    unit = 2.0 ** (-8 - 8 * np.arange(3))
    P.eri_tttc = np.full_like(P.eri_tttc, dx @ unit)
    P.groups[0].ci = np.eye(len(dets))
    row = coracle.Oracle(P).class4_rows(0, 1).reshape(len(dets), n_co)[:, 0]
    assert np.all(np.abs(row) == dx @ unit)
    P.groups[0].ci = np.ascontiguousarray((np.sign(row) * (dc @ unit))[:, None])
    products = [int(sum((dx[i] * dc[:, s - i]).sum() for i in range(s + 1))) << (16 - 8 * s) for s in range(3)]
    return P, sum(products) * 2.0 ** -32


def test_coherent_digits():
    """Three slices: the six products of a term that are formed are summed exactly."""
    import torch
    from paper_1709_03005_gb300 import hb
    P, want = _coherent_terms()
    H = hb.Hamiltonian(P, class4_path=2, split_slices=3)
    b, _ = H.build(hb.HB_MIXED)
    torch.cuda.synchronize()
    assert "class4 tensor cores" in H.tuning_report()
    got = b["Hlc"].cpu().numpy()
    H.close()
    assert np.array_equal(got, np.full_like(got, want)), (got - want) * 2.0 ** 32

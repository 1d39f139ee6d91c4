"""Contexts that borrow their integrals (hb_init_shared): what the base must
have, and what becomes of the borrowed tables."""
import pytest

from paper_1709_03005_gb300 import synth

pytestmark = pytest.mark.gpu
KEYS = ("Hcc", "Hlc", "row_ptr", "col", "val")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


def _base_and_problem():
    """A base problem and another one over its integrals."""
    base = synth.make_config("mid")
    P = synth.make_config("mid", n_state=5, n_l2=150, seed=11)
    for name in ("h", "eri_tttt", "eri_tttc", "eri_ttcc", "eri_tctc"):
        setattr(P, name, getattr(base, name))
    return base, P


def _reference(P, precision):
    import torch
    from paper_1709_03005_gb300 import hb
    H = hb.Hamiltonian(P)
    b, _ = H.build(precision)
    torch.cuda.synchronize()
    H.close()
    return b


def test_base_without_groups():
    """It holds no continuum integrals: target groups cannot borrow from it, L2 functions alone can."""
    import torch
    from paper_1709_03005_gb300 import hb
    base, P = _base_and_problem()
    base.groups = []
    B = hb.Hamiltonian(base)
    with pytest.raises(hb.HBError) as e:
        hb.Hamiltonian(P, base=B)
    assert e.value.code == hb.HB_ERR_INVALID_ARG
    P.groups = []
    ref = _reference(P, 0)
    H = hb.Hamiltonian(P, base=B)
    b, _ = H.build(0)
    torch.cuda.synchronize()
    for k in ("row_ptr", "col", "val"):
        assert torch.equal(b[k], ref[k]), k
    H.close()
    B.close()

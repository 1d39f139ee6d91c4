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


@pytest.mark.parametrize("precision", [0, 1])
def test_tables_made_on_another_stream(precision):
    """The first build of a borrowing context, on another stream, beside the base's
    first build (or contraction) that makes the tables and is held up ahead of them."""
    import torch
    from paper_1709_03005_gb300 import hb
    base, P = _base_and_problem()
    ref = _reference(P, precision)
    B = hb.Hamiltonian(base)
    H = hb.Hamiltonian(P, base=B)
    out = H.allocate()
    x, part = B.allocate(), torch.empty(B.shard_coef_len(), dtype=torch.float64, device="cuda")
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(a):
        torch.cuda._sleep(400_000_000)          # 0.2 s
        if precision == 0:
            B.build(0, x, stream=a, stats=False)
        else:
            B.build_contract(1, 0, 1, part, stream=a)
    H.build(precision, out, stream=b, stats=False)
    b.synchronize()
    for k in KEYS:
        assert torch.equal(out[k], ref[k]), k
    torch.cuda.synchronize()
    H.close()
    B.close()

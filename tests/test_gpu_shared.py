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


def _overwrite_freed():
    """Fill what the device has just been given back with NaN patterns."""
    import torch
    x = [torch.full((1 << 20,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(64)]
    torch.cuda.synchronize()
    del x


@pytest.mark.parametrize("precision", [0, 1])
def test_tables_released_by_the_base(precision):
    """The base measures and takes a workspace, which releases the tables it had
    lent: the borrowing context's builds, replayed ones too, do not read them any more."""
    import torch
    from paper_1709_03005_gb300 import hb
    base, P = _base_and_problem()
    ref, ref_base = _reference(P, precision), _reference(base, precision)
    B = hb.Hamiltonian(base)
    H = hb.Hamiltonian(P, base=B)
    out = H.allocate()
    for _ in range(4):
        H.build(precision, out)
    need = B.workspace_size(precision)
    _overwrite_freed()
    out["Hcc"].fill_(0.0)
    H.build(precision, out)
    torch.cuda.synchronize()
    for k in KEYS:
        assert torch.equal(out[k], ref[k]), k
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    B.set_workspace(ws)
    _overwrite_freed()
    x, _ = B.build(precision)
    out["Hcc"].fill_(0.0)
    H.build(precision, out)
    torch.cuda.synchronize()
    for k in KEYS:
        assert torch.equal(out[k], ref[k]) and torch.equal(x[k], ref_base[k]), k
    H.close()
    B.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_tables_of_a_batch_stay(precision):
    """Members of a batch measure and take a workspace: the batch's graph still reads their tables."""
    import torch
    from paper_1709_03005_gb300 import hb
    base, P = _base_and_problem()
    B = hb.Batch([base, P], precision)
    B.launch()
    torch.cuda.synchronize()
    ref = [{k: v.clone() for k, v in b.items()} for b in B.blocks]
    ws = []
    for h in B.hams:
        ws.append(torch.empty(h.workspace_size(precision), dtype=torch.uint8, device="cuda"))
        h.set_workspace(ws[-1])
    _overwrite_freed()
    for b in B.blocks:
        b["Hcc"].fill_(0.0)
    B.launch()
    torch.cuda.synchronize()
    for b, r in zip(B.blocks, ref):
        for k in KEYS:
            assert torch.equal(b[k], r[k]), k
    for h, r in zip(B.hams, ref):
        b, _ = h.build(precision)
        torch.cuda.synchronize()
        for k in KEYS:
            assert torch.equal(b[k], r[k]), k
    B.close()

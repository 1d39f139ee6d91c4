"""Contexts of different split_slices that meet in one plan: a context that
borrows its integrals takes the class-4 slices of the context that owns them,
whichever of the two is built first; batches of different counts are refused,
and those of the same class-4 count but different expansion digits (6 given, and
the default) are accepted."""
import ctypes as C

import pytest

from paper_1709_03005_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


def _problem():
    return synth.make_config("mid", n_co=20, n_state=36, n_l2=60, seed=77)


def _build(H):
    import torch
    from paper_1709_03005_gb300 import hb
    b, _ = H.build(hb.HB_MIXED)
    torch.cuda.synchronize()
    return b


@pytest.mark.parametrize("base_first", [True, False])
@pytest.mark.parametrize("base_slices,slices", [(4, 0), (0, 3), (3, 5)])
def test_borrowed_integrals(base_slices, slices, base_first):
    import torch
    from paper_1709_03005_gb300 import hb
    P = _problem()
    want = hb.Hamiltonian(P, split_slices=base_slices)
    ref = _build(want)
    base = hb.Hamiltonian(P, split_slices=base_slices)
    H = hb.Hamiltonian(P, split_slices=slices, base=base)
    order = [base, H] if base_first else [H, base]
    for h in order + order:
        b = _build(h)
        assert "class4 tensor cores" in h.tuning_report()
        for k in ("Hcc", "Hlc", "val"):
            assert torch.equal(b[k], ref[k]), k
    for h in (H, base, want):
        h.close()


def _batch(hams, precision):
    from paper_1709_03005_gb300 import hb
    lib = hb.load()
    blocks = [h.allocate() for h in hams]
    ctxs = (C.c_void_p * len(hams))(*[h.ctx.value for h in hams])
    outs = (hb.hb_blocks * len(hams))(*[hb.Hamiltonian.blocks_struct(b) for b in blocks])
    handle = C.c_void_p()
    lib.hb_batch_create.argtypes = [C.POINTER(C.c_void_p), C.c_void_p, C.c_int32, C.c_int32, C.c_void_p, C.c_void_p]
    lib.hb_batch_destroy.argtypes = [C.c_void_p]
    lib.hb_batch_destroy.restype = None
    return lib, lib.hb_batch_create(C.byref(handle), ctxs, len(hams), precision, outs, None), handle, blocks


@pytest.mark.parametrize("a,b,accepted", [(5, 0, False), (4, 3, False), (6, 0, True), (0, 0, True)])
def test_batches(a, b, accepted):
    import torch
    from paper_1709_03005_gb300 import hb
    P = _problem()
    hams = [hb.Hamiltonian(P, split_slices=a), hb.Hamiltonian(P, split_slices=b)]
    lib, rc, handle, blocks = _batch(hams, hb.HB_MIXED)
    assert rc == (hb.HB_OK if accepted else hb.HB_ERR_INVALID_ARG)
    if accepted:
        lib.hb_batch_launch.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p]
        assert lib.hb_batch_launch(handle, None, None) == hb.HB_OK
        torch.cuda.synchronize()
        for h, got in zip(hams, blocks):
            ref = _build(h)
            assert torch.equal(got["Hlc"], ref["Hlc"]) and torch.equal(got["val"], ref["val"])
            # the leading digits of a longer expansion: the same bound, not the same bits
            tol = 1e-11 * ref["Hcc"].abs().max()
            assert (got["Hcc"] - ref["Hcc"]).abs().max() <= tol
        lib.hb_batch_destroy(handle)
        # FP64 builds have no such choice
    lib, rc, handle, blocks = _batch(hams, hb.HB_FP64)
    assert rc == hb.HB_OK
    lib.hb_batch_destroy(handle)
    for h in hams:
        h.close()


def test_base_without_a_wide_group():
    """A base context none of whose groups takes class 4 on the tensor cores lends the tables all the same."""
    import torch
    from paper_1709_03005_gb300 import hb
    P = _problem()
    narrow = synth.make_config("mid", n_co=20, n_state=3, n_l2=60, seed=77)
    for name in ("h", "eri_tttt", "eri_tttc", "eri_ttcc", "eri_tctc"):
        setattr(narrow, name, getattr(P, name))
    want = hb.Hamiltonian(P)
    ref = _build(want)
    base = hb.Hamiltonian(narrow)
    _build(base)
    H = hb.Hamiltonian(P, base=base)
    b = _build(H)
    assert "class4 tensor cores" in H.tuning_report()
    for k in ("Hcc", "Hlc", "val"):
        assert torch.equal(b[k], ref[k]), k
    _build(base)
    for h in (H, base, want):
        h.close()

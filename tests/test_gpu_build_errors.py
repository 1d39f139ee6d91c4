"""A wait that gave up in a build, set by a test hook: the call that learns of it
returns HB_ERR_TIMEOUT once, whatever the precision, and the build after it runs."""
import ctypes as C

import pytest

from paper_1709_03005_gb300 import synth

pytestmark = pytest.mark.gpu
KEYS = ("Hcc", "Hlc", "row_ptr", "col", "val")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


def _inject(H, word, following):
    H.lib.hb_test_build_error.argtypes = [C.c_void_p, C.c_int, C.c_int]
    assert H.lib.hb_test_build_error(H.ctx, word, following) == 0


def _times_out(call):
    from paper_1709_03005_gb300 import hb
    with pytest.raises(hb.HBError) as e:
        call()
    assert e.value.code == hb.HB_ERR_TIMEOUT


def _same(a, b):
    import torch
    torch.cuda.synchronize()
    for k in KEYS:
        assert torch.equal(a[k], b[k]), k


def test_mixed_build_is_told_once():
    from paper_1709_03005_gb300 import hb
    H = hb.Hamiltonian(synth.make_config("c1"))
    ref, _ = H.build(1)
    x = H.allocate()
    for _ in range(3):
        _inject(H, 5, 1)
        _times_out(lambda: H.build(1, x))
        H.build(1, x)
        _same(x, ref)
    H.close()


@pytest.mark.parametrize("waits", [True, False])
def test_fp64_build_is_told_once(waits):
    """With stats the call itself waits and tells, without them the next build."""
    from paper_1709_03005_gb300 import hb
    H = hb.Hamiltonian(synth.make_config("c1"))
    ref, _ = H.build(0)
    x = H.allocate()
    for _ in range(3):
        _inject(H, 5, 1)
        if waits:
            _times_out(lambda: H.build(0, x))
        else:
            H.build(0, x, stats=False)
            _times_out(lambda: H.build(0, x, stats=False))
        H.build(0, x, stats=False)
        _same(x, ref)
    H.close()


def test_batch_is_told_once():
    from paper_1709_03005_gb300 import hb
    B = hb.Batch([synth.make_config("c1")], 1)
    H = B.hams[0]
    B.launch()
    ref = {k: v.clone() for k, v in B.blocks[0].items()}
    _inject(H, 5, 1)
    _times_out(B.launch)
    x, _ = H.build(1)                   # the batch has told it
    _same(x, ref)
    B.launch()
    _same(B.blocks[0], ref)
    B.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_shard_is_told_once(precision):
    from paper_1709_03005_gb300 import hb
    H = hb.Hamiltonian(synth.make_config("c1"))
    red, _ = H.build_contract(precision, 0, 1)
    red = red.clone()
    ref, _ = H.build_expand(precision, 0, 1, red)
    x = H.allocate()
    _inject(H, 5, 1)
    if precision:
        _times_out(lambda: H.build_expand(precision, 0, 1, red, x))
    else:
        H.build_expand(precision, 0, 1, red, x)
        _times_out(lambda: H.build_contract(precision, 0, 1))
    H.build_contract(precision, 0, 1)
    H.build_expand(precision, 0, 1, red, x)
    _same(x, ref)
    H.close()


def test_solve_after_a_failed_fp64_build():
    from paper_1709_03005_gb300 import hb
    H = hb.Hamiltonian(synth.make_config("c1"))
    x, _ = H.build(0)
    ref, _, _ = H.diag(x, 2)
    for flags in (hb.HB_PRECOND_DIAG, hb.HB_PRECOND_DIAG | hb.HB_DIAG_TENSOR):
        _inject(H, 5, 1)
        H.build(0, x, stats=False)
        _times_out(lambda: H.diag(x, 2, precond=flags))
        ev, _, _ = H.diag(x, 2)
        assert (ev == ref).all()
    H.close()


def test_change_of_precision_after_a_failed_fp64_build():
    from paper_1709_03005_gb300 import hb
    H = hb.Hamiltonian(synth.make_config("c1"))
    ref, _ = H.build(1)
    x, _ = H.build(0)
    _inject(H, 5, 1)
    H.build(0, x, stats=False)
    _times_out(lambda: H.build(1, x))
    H.build(1, x)
    _same(x, ref)
    H.close()


def test_fp64_batch_that_waits():
    from paper_1709_03005_gb300 import hb
    B = hb.Batch([synth.make_config("c1")], 0)
    B.launch()
    ref = {k: v.clone() for k, v in B.blocks[0].items()}
    _inject(B.hams[0], 5, 1)
    _times_out(B.launch)
    B.launch()
    _same(B.blocks[0], ref)
    B.close()

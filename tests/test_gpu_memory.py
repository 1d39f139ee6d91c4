"""Device memory of the tables made on first use: what a failed set-up leaves, and
what an FP64 build takes."""
import ctypes as C

import pytest

from paper_1709_03005_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


def test_failed_setup_holds_nothing():
    """A workspace that takes the panel slices of a mixed build and no more: every
    attempt fails alike, and none of them keeps the slices."""
    import torch
    from paper_1709_03005_gb300 import hb
    P = synth.make_config("mid")
    H = hb.Hamiltonian(P)
    L = H.layout
    Kc = (L.n_labels + 63) // 64 * 64
    slices = 5 * 2 * P.n_co ** 2 * Kc
    H.set_workspace(torch.empty(slices + 4096, dtype=torch.uint8, device="cuda"))
    held = L.device_bytes
    seen = set()
    for _ in range(3):
        with pytest.raises(hb.HBError) as e:
            H.build(hb.HB_MIXED)
        assert e.value.code == hb.HB_ERR_OOM
        seen.add(str(e.value))
        hb._check(H.lib.hb_query(H.ctx, C.byref(L)), H.ctx)
        assert L.device_bytes == held
    assert len(seen) == 1
    H.close()


def test_solve_after_one_without_room():
    """A workspace for a solve of 2 pairs: one of 24 finds no room, the next of 2 runs as before."""
    import numpy as np
    import torch
    from paper_1709_03005_gb300 import hb
    H = hb.Hamiltonian(synth.make_config("mid"))
    x, _ = H.build(0)
    need = H.workspace_size(-1, 2) - (14 << 20)      # most of its allowance for the autotuner
    H.set_workspace(torch.empty(need, dtype=torch.uint8, device="cuda"))
    ref, _, _ = H.diag(x, 2)
    for _ in range(2):
        with pytest.raises(hb.HBError) as e:
            H.diag(x, 24)
        assert e.value.code == hb.HB_ERR_OOM
        ev, _, _ = H.diag(x, 2)
        assert np.array_equal(ev, ref)
    H.close()


def _fill_device_but(left):
    """Take all device memory but about `left` bytes."""
    import torch
    torch.cuda.empty_cache()
    return torch.empty(max(torch.cuda.mem_get_info()[0] - left, 0), dtype=torch.uint8, device="cuda")


def test_error_of_an_allocation_is_returned_once():
    """A solve that finds no memory; what follows it with room again succeeds."""
    import numpy as np
    import torch
    from paper_1709_03005_gb300 import hb
    P = synth.make_config("c2")
    H = hb.Hamiltonian(P)
    x, _ = H.build(1)
    rest = _fill_device_but(64 << 20)
    with pytest.raises(hb.HBError) as e:
        H.diag(x, 20, 1e-6)
    assert e.value.code == hb.HB_ERR_OOM
    with pytest.raises(hb.HBError) as e:
        hb.Hamiltonian(P)
    assert e.value.code == hb.HB_ERR_OOM
    del rest
    torch.cuda.empty_cache()
    ev, _, _ = H.diag(x, 20, 1e-6)
    G = hb.Hamiltonian(P)
    y, _ = G.build(1)
    assert torch.equal(x["Hcc"], y["Hcc"])
    assert np.isfinite(ev).all()
    G.close()
    H.close()


def _build64(H, x=None):
    import torch
    b, st = H.build(0, x)
    torch.cuda.synchronize()
    return b, st


def test_fp64_slices_take_a_quarter_of_the_free_memory():
    """0.51 GB of slices beside 1.5 GB of free memory: the build adds its sums on the FP64 pipe, and holds no more than it did."""
    import torch
    from paper_1709_03005_gb300 import hb
    P = synth.make_config("c2")
    H = hb.Hamiltonian(P)
    x = H.allocate()
    rest = _fill_device_but(3 << 29)
    before = torch.cuda.mem_get_info()[0]
    _, st = _build64(H, x)
    assert st.expand_tensor_flops == 0.0
    assert before - torch.cuda.mem_get_info()[0] < 64 << 20
    want = {k: v.clone() for k, v in x.items()}
    del rest
    torch.cuda.empty_cache()
    H.close()
    H = hb.Hamiltonian(P)
    _, st = _build64(H, x)
    assert st.expand_tensor_flops > 0.0
    scale = want["Hcc"].abs().max()
    assert (x["Hcc"] - want["Hcc"]).abs().max() <= 1e-13 * scale
    assert torch.equal(x["Hlc"], want["Hlc"]) and torch.equal(x["val"], want["val"])
    H.close()


@pytest.mark.parametrize("what", ["solve", "mixed"])
def test_fp64_slices_are_given_back(what):
    """What finds no room beside the slices of an earlier FP64 build takes theirs."""
    import numpy as np
    import torch
    from paper_1709_03005_gb300 import hb
    P = synth.make_config("c2")
    H = hb.Hamiltonian(P)
    if what == "solve":
        x, _ = _build64(H)
        ref, _, _ = H.diag(x, 20, 1e-6)
    else:
        x, _ = H.build(1)
        ref = {k: v.clone() for k, v in x.items()}
    H.close()
    H = hb.Hamiltonian(P)
    _, st = _build64(H, x)
    assert st.expand_tensor_flops > 0.0
    y = torch.zeros_like(x["Hcc"])
    rest = _fill_device_but(128 << 20)
    if what == "solve":
        ev, _, _ = H.diag(x, 20, 1e-6)
        assert np.array_equal(ev, ref)
    else:
        H.build(1, x)
        torch.cuda.synchronize()
        for k in ref:
            assert torch.equal(x[k], ref[k]), k
    _build64(H, x)
    del rest, y
    torch.cuda.empty_cache()
    H.close()


def test_scratch_of_many_roots():
    """200 roots of dimension 959 (up to 959 vectors): the partial sums of the
    projections take no more than the vectors do, and the solve is right."""
    import numpy as np
    import torch
    from oracle import coracle
    from paper_1709_03005_gb300 import hb
    P = synth.make_config("mid")
    H = hb.Hamiltonian(P)
    need = H.workspace_size(-1, 200)
    vectors = 5 * 8 * H.dim * H.dim
    assert need <= 3 * vectors
    x, _ = _build64(H)
    H.set_workspace(torch.empty(need, dtype=torch.uint8, device="cuda"))
    ev, _, _ = H.diag(x, 200, 1e-8, 200)
    ref = np.linalg.eigvalsh(coracle.Oracle(P).dense())[:200]
    np.testing.assert_allclose(ev, ref, atol=1e-8, rtol=0)
    H.close()

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

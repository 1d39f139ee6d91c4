"""Builds repeated into the same blocks (replayed as a graph from the third
on), with other blocks, another stream and the other precision in between:
every build writes everything again, to the same bits, with its stage times."""
import pytest

from paper_1709_03005_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


def _clear(b):
    for k in ("Hcc", "Hlc", "val"):
        b[k].fill_(float("nan"))
    for k in ("row_ptr", "col"):
        b[k].fill_(-1)


@pytest.mark.parametrize("key", ["c1", "mid"])
def test_repeated_builds(key):
    import torch
    from paper_1709_03005_gb300 import hb
    H = hb.Hamiltonian(synth.make_config(key))
    ref = {}
    for p in (hb.HB_FP64, hb.HB_MIXED):
        ref[p], _ = H.build(p)
    first, other = H.allocate(), H.allocate()
    side = torch.cuda.Stream()
    for p in (hb.HB_MIXED, hb.HB_FP64):
        for blocks, stream in [(first, None)] * 5 + [(other, None)] * 2 + [(first, side)] * 5 + [(other, side)] * 4:
            _clear(blocks)
            torch.cuda.synchronize()
            _, st = H.build(p, blocks, stream=stream)
            torch.cuda.synchronize()
            assert st.ms_total > 0 and st.ms_target > 0 and st.kernel_launches > 10
            for k in ref[p]:
                assert torch.equal(blocks[k], ref[p][k]), (p, k)
    # without stats the FP64 build does not wait: several may be in flight
    for _ in range(6):
        _clear(first)
        for _ in range(3):
            H.build(hb.HB_FP64, first, stats=False)
    torch.cuda.synchronize()
    for k in ref[hb.HB_FP64]:
        assert torch.equal(first[k], ref[hb.HB_FP64][k]), k
    H.close()

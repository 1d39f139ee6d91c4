"""Builds of one context enqueued on different streams without waiting in
between: each runs behind the one before, whichever of the two was launched
directly, replayed as a graph, part of a batch or a shard.  The first stream is
held up ahead of its build; when the second stream has finished, that build must
be done, and both blocks must hold the matrix."""
import pytest

from paper_1709_03005_gb300 import synth

pytestmark = pytest.mark.gpu
KEYS = ("Hcc", "Hlc", "row_ptr", "col", "val")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


def _ordered(first, second):
    """first(stream) behind a long wait on one stream, second(stream) on another: the first is done when the second is."""
    import torch
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    with torch.cuda.stream(a):
        torch.cuda._sleep(400_000_000)          # 0.2 s
        first(a)
        done.record(a)
    second(b)
    b.synchronize()
    assert done.query(), "the second build did not wait for the first"
    torch.cuda.synchronize()


@pytest.mark.parametrize("before", [0, 1, 3], ids=["direct", "then-replay", "replay"])
@pytest.mark.parametrize("other_blocks", [False, True])
def test_own_builds(before, other_blocks):
    import torch
    from paper_1709_03005_gb300 import hb
    H = hb.Hamiltonian(synth.make_config("c1"))
    ref, _ = H.build(0)
    torch.cuda.synchronize()
    x, y = H.allocate(), H.allocate()
    for _ in range(before):
        H.build(0, x, stats=False)
    z = y if other_blocks else x
    _ordered(lambda s: H.build(0, x, stream=s, stats=False), lambda s: H.build(0, z, stream=s, stats=False))
    for k in KEYS:
        assert torch.equal(ref[k], x[k]) and torch.equal(ref[k], z[k]), k
    H.close()


def test_batch_and_own_build():
    import torch
    from paper_1709_03005_gb300 import hb
    B = hb.Batch([synth.make_config("c1")], precision=0)
    H, x = B.hams[0], B.hams[0].allocate()
    ref, _ = H.build(0)
    H.build(0, x, stats=False)
    _ordered(lambda s: B.launch(stream=s, stats=False), lambda s: H.build(0, x, stream=s, stats=False))
    _ordered(lambda s: H.build(0, x, stream=s, stats=False), lambda s: B.launch(stream=s, stats=False))
    for k in KEYS:
        assert torch.equal(ref[k], x[k]), k
    B.close()


def test_shard_and_own_build():
    import torch
    from paper_1709_03005_gb300 import hb
    H = hb.Hamiltonian(synth.make_config("c1"))
    ref, _ = H.build(0)
    part, _ = H.build_contract(0, 0, 1)
    want = part.clone()
    x = H.allocate()
    H.build(0, x, stats=False)
    _ordered(lambda s: H.build(0, x, stream=s, stats=False), lambda s: H.build_contract(0, 0, 1, part, stream=s))
    assert torch.equal(part, want)
    for k in KEYS:
        assert torch.equal(ref[k], x[k]), k
    H.close()

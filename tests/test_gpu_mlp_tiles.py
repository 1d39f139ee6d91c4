"""The training kernel at the edges of its sample tiles (128 samples) and of
the grid (a block per SM): loss and gradient against the FP64 reference."""
import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


@pytest.mark.parametrize("n", [1, 3, 127, 128, 129, 152 * 128, 152 * 128 + 1, 40001])
def test_gradient_at_tile_edges(n):
    """Every sum has at most 72 terms per sample and n / 152 + 152 additions in
    a row over samples, each rounded to 2^-24: below 1e-4 of the largest
    gradient at these sizes (the bound the whole-network test uses).  Samples
    after the last are poisoned: they must not be read."""
    import torch
    from paper_1709_03005_gb300 import hb
    rng = np.random.default_rng(n)
    p = rng.normal(0, 0.2, 4801).astype(np.float32)
    f = rng.normal(0, 1, (n, 8)).astype(np.float32)
    a, b = rng.normal(0, 1, (2, n)).astype(np.float32)
    pad = lambda x: torch.from_numpy(np.concatenate([x, np.full((256,) + x.shape[1:], np.nan, np.float32)])).cuda()[:n]
    loss, g = hb.mlp_loss_grad(torch.from_numpy(p).cuda(), pad(f), pad(a), pad(b))
    torch.cuda.synchronize()
    ref_loss, ref_g = mlp.loss_grad(p.astype(np.float64), f.astype(np.float64), a.astype(np.float64),
                                    b.astype(np.float64))
    assert abs(float(loss) - ref_loss) <= 1e-5 * abs(ref_loss)
    np.testing.assert_allclose(g.cpu().numpy(), ref_g, rtol=1e-3, atol=1e-4 * np.abs(ref_g).max())

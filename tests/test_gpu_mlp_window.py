"""Training gradients over a window far beyond the default: the FP32 sums over the
samples are chains of at most 1024 additions, whatever the window."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


def test_equal_samples():
    """Five million copies of one sample, 256 tiles a block: the mean of their
    gradients is the sample's.  A sum of equal terms is off by half an ulp of what it
    has reached at most, every time with the same sign: 1024 additions, then 32 sums of
    such, 152 blocks in eights and three of the reduction, each rounded to 2^-24."""
    import torch
    from paper_1709_03005_gb300 import hb
    n = 256 * 152 * 128
    rng = np.random.default_rng(5)
    p = torch.tensor(rng.normal(0, 0.2, 4801), dtype=torch.float32, device="cuda")
    f = torch.tensor(rng.normal(0, 1, (1, 8)), dtype=torch.float32, device="cuda")
    a, b = (torch.tensor([v], dtype=torch.float32, device="cuda") for v in (0.7, -0.4))
    loss1, g1 = hb.mlp_loss_grad(p, f, a, b)
    loss, g = hb.mlp_loss_grad(p, f.repeat(n, 1), a.repeat(n), b.repeat(n))
    torch.cuda.synchronize()
    off = ((g.double() - g1.double()).abs() / g1.double().abs())[g1 != 0.0].max().item()
    assert torch.equal(g[g1 == 0.0], g1[g1 == 0.0])
    assert off <= (1024 + 32 + 19 + 8 + 3) * 2.0 ** -24, off
    assert abs(float(loss) / float(loss1) - 1.0) <= (256 + 19 + 18) * 2.0 ** -24

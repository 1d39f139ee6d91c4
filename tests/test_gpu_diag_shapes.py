"""Davidson's vector kernels at the edges of their tiles: block widths below,
at and beyond 16 and 32 vectors, matrices of a few rows and of several product
slices; eigenvalues and residuals against the dense FP64 eigensolver."""
import numpy as np
import pytest

from oracle import coracle
from paper_1709_03005_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


@pytest.mark.parametrize("key,over,ks", [("mid", {}, (1, 11, 12, 24, 45)), ("c1", dict(n_l2=0), (1, 7)),
                                         ("mid", dict(n_l2=1, n_co=17), (3, 20))])
def test_eigenpairs(key, over, ks):
    import torch
    from paper_1709_03005_gb300 import hb
    P = synth.make_config(key, **over)
    R = coracle.Oracle(P).dense()
    ref = np.linalg.eigvalsh(R)
    H = hb.Hamiltonian(P)
    b, _ = H.build(hb.HB_FP64)
    for k in ks:
        for flags in (0, hb.HB_DIAG_TENSOR):
            X = torch.zeros((P.dim, k), dtype=torch.float64, device="cuda")
            w, _, _ = H.diag(b, k, 1e-8, 500, precond=hb.HB_PRECOND_DIAG | flags, evecs=X)
            torch.cuda.synchronize()
            np.testing.assert_allclose(w, ref[:k], atol=1e-8, rtol=0)
            x = X.cpu().numpy()
            assert np.linalg.norm(R @ x - x * w, axis=0).max() <= 1e-8 * 1.01
            np.testing.assert_allclose(x.T @ x, np.eye(k), atol=1e-10)
    H.close()

"""FP64 builds whose rows of labels have a wide range: the largest entries of the
panel row meet zeros of the coefficient row, or the other way round, so that the
terms are far below the scales of the digit slices.  Every element is as close to
the oracle as sums in FP64 are, |G - R| <= 64 u sum |terms|.  An infinity or a NaN
of such a row spreads as it does in those sums."""
import numpy as np
import pytest

from gpu_util import FP64_FALLBACK
from oracle import coracle
from paper_1709_03005_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


def _pair(p, q):
    return p * (p + 1) // 2 + q


def _large_h(h, eri):
    """Two groups that share no determinant, S = 0 between them: h_jj' sets the scale and adds nothing."""
    P = synth.make_config("mid", n_to=10, n_co=19, n_det=40, n_state=[3, 2], n_l2=0, n_groups=2, seed=21)
    c = slice(P.n_to, None)
    P.h[c, c] *= h / np.abs(P.h[c, c]).max()
    P.eri_ttcc *= eri
    P.eri_tctc *= eri
    return P


def _unused_orbital(scale):
    """No determinant holds the last target orbital, whose integrals are the largest."""
    P = synth.make_config("mid", n_to=10, n_co=19, n_det=40, n_state=4, n_l2=0, seed=22)
    P.groups = synth.make_config("mid", n_to=9, n_co=19, n_det=40, n_state=4, n_l2=0, seed=22).groups
    t, nt, nc = P.n_to - 1, P.n_to, P.n_co
    P.eri_ttcc[[_pair(t, q) for q in range(nt)]] *= scale
    x = P.eri_tctc.reshape(nt, nc, nt, nc)
    x[t] *= scale
    x[:, :, t] *= scale
    return P


def _small_mixing(mix):
    """The reference with a small admixture; integrals of its occupied pairs are zero:
    the large densities meet zeros."""
    P = synth.make_config("mid", n_to=10, n_co=19, n_det=40, n_state=2, n_l2=0, seed=23)
    g = P.groups[0]
    rng = np.random.default_rng(1)
    # the reference is among the determinants: the lowest orbitals of both spins
    half = P.n_elec // 2
    ref = int(np.nonzero((g.dets == (1 << half) - 1).all(1))[0][0])
    ci = mix * rng.standard_normal(g.ci.shape)
    ci[ref] = 1.0
    g.ci = ci
    nt, nc = P.n_to, P.n_co
    P.eri_ttcc[[_pair(p, q) for p in range(half) for q in range(p + 1)]] = 0.0
    x = P.eri_tctc.reshape(nt, nc, nt, nc)
    x[:half, :, :half] = 0.0
    off = ~np.eye(nc, dtype=bool)
    P.h[nt:, nt:][off] = 0.0
    return P


CASES = dict(h10=lambda: _large_h(10.0, 1e-4), h50=lambda: _large_h(50.0, 1e-6), h_far=lambda: _large_h(1.0, 1e-30),
             unused=lambda: _unused_orbital(1e7), unused_far=lambda: _unused_orbital(1e40),
             mixing=lambda: _small_mixing(1e-6), subnormal=lambda: _large_h(1.0, 1e-310))


def _hcc(P, **kw):
    import torch
    from paper_1709_03005_gb300 import hb
    H = hb.Hamiltonian(P, **kw)
    b, st = H.build(0)
    torch.cuda.synchronize()
    assert st.expand_tensor_flops > 0.0
    out = b["Hcc"].cpu().numpy()
    H.close()
    return out


@pytest.mark.parametrize("name", list(CASES))
def test_wide_rows(name):
    P = CASES[name]()
    o = coracle.Oracle(P)
    G, R, S = _hcc(P), o.dense(), o.condition()
    d = np.abs(G - R)
    # and what underflows: 157 labels, a product and a sum each, on either side
    bound = FP64_FALLBACK * S + 157 * 4 * 2.5e-324
    assert (d <= bound).all(), (d / np.maximum(bound, 1e-320)).max()
    assert np.array_equal(G, G.T)
    for cols in (32, 64):
        for tile in (3, 4, 5):
            assert np.array_equal(_hcc(P, split_cols=cols, split_tile=tile), G), (cols, tile)

"""The expansion's digit slices where they can go wrong: rows whose digits are
all large and of one sign (every accumulator then reaches its exact span), tile
widths and ragged columns of the FP64 kernel, values that are not finite, rows
far from 1 in magnitude, and the FP64 sums that take over when the slices have
no room."""
import numpy as np
import pytest

from gpu_util import FP64_FALLBACK, MIXED_CC_FALLBACK, check_elements
from oracle import coracle
from paper_1709_03005_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


def _build(P, precision, **kw):
    import torch
    from paper_1709_03005_gb300 import hb
    H = hb.Hamiltonian(P, validate=False, **kw)
    b, _ = H.build(precision)
    torch.cuda.synchronize()
    out = b["Hcc"].cpu().numpy()
    H.close()
    return out


def _coherent(sign):
    """Every two-electron integral of the continuum classes is the same number
    (of both signs alternately for sign < 0), whose base-512 digits are all 255:
    the slice products of a row add up without cancelling."""
    P = synth.make_problem("digits", 5, 20, 9, 6, 30, 5, 0, 8)
    x = sum(255.0 * 2.0 ** (-8 - 9 * i) for i in range(6))
    P.eri_ttcc = np.full_like(P.eri_ttcc, x)
    P.eri_tctc = np.full_like(P.eri_tctc, sign * x)
    for g in P.groups:
        g.ci = np.ascontiguousarray(np.abs(g.ci))
    return P


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("precision", [0, 1])
def test_coherent_digits(precision, sign):
    P = _coherent(sign)
    o = coracle.Oracle(P)
    check_elements(_build(P, precision), o.dense(), o.condition(), (1e-12, 1e-10)[precision],
                   (FP64_FALLBACK, MIXED_CC_FALLBACK)[precision], "coherent digits")


@pytest.mark.parametrize("kw", [dict(n_state=1), dict(n_state=7), dict(n_state=8, n_co=17), dict(n_state=11, n_co=33)])
def test_fp64_tile_widths(kw):
    """28, 36 and 66 state pairs: one and several tiles of 32 and 64 columns give the same bits."""
    P = synth.make_config("mid", n_l2=5, **kw)
    o = coracle.Oracle(P)
    ref = _build(P, 0)
    check_elements(ref[: o.Dc, : o.Dc], o.dense()[: o.Dc, : o.Dc], o.condition()[: o.Dc, : o.Dc], 1e-12, FP64_FALLBACK,
                   "FP64 tiles")
    for cols in (32, 64, 128):
        for tile in (3, 4, 5):
            assert np.array_equal(_build(P, 0, split_cols=cols, split_tile=tile), ref), (cols, tile)


@pytest.mark.parametrize("scale", [2.0 ** -200, 2.0 ** 150])
def test_fp64_scaled_integrals(scale):
    """Powers of two scale the whole matrix exactly: the row exponents are kept apart from the digits."""
    P = synth.make_config("c1", n_l2=0)
    ref = _build(P, 0)
    for name in ("h", "eri_tttt", "eri_tttc", "eri_ttcc", "eri_tctc"):
        setattr(P, name, getattr(P, name) * scale)
    assert np.array_equal(_build(P, 0), ref * scale)


def test_fp64_not_finite():
    """A NaN or an infinity among the integrals of one continuum pair reaches every element of that pair and no other."""
    P = synth.make_config("c1", n_l2=0)
    ref = _build(P, 0)
    nan, inf = (3, 7), (1, 4)
    for (j, k), v in ((nan, np.nan), (inf, np.inf)):
        P.eri_ttcc[2, j * P.n_co + k] = P.eri_ttcc[2, k * P.n_co + j] = v
    G = _build(P, 0)
    bad = np.zeros((P.n_co, P.n_co), bool)
    for j, k in (nan, inf):
        bad[j, k] = bad[k, j] = True
    ns = P.groups[0].ci.shape[1]
    bad = np.tile(bad, (ns, ns))
    assert not np.isfinite(G[bad]).any()
    assert np.array_equal(G[~bad], ref[~bad])


def test_fp64_without_room_for_slices():
    """A workspace that was not sized for an FP64 build: the sums run on the
    FP64 pipe, in the memory such a build always took, and agree to rounding."""
    import torch
    from paper_1709_03005_gb300 import hb
    P = synth.make_config("mid")
    o = coracle.Oracle(P)
    ref = _build(P, 0)
    H = hb.Hamiltonian(P)
    ws = torch.empty(H.workspace_size(hb.HB_MIXED), dtype=torch.uint8, device="cuda")
    H.set_workspace(ws)
    b, st = H.build(hb.HB_FP64)
    torch.cuda.synchronize()
    assert st.expand_tensor_flops == 0.0
    G = b["Hcc"].cpu().numpy()
    H.close()
    R, S = o.dense()[: o.Dc, : o.Dc], o.condition()[: o.Dc, : o.Dc]
    check_elements(G, R, S, 1e-12, FP64_FALLBACK, "FP64 pipe")
    check_elements(ref, R, S, 1e-12, FP64_FALLBACK, "FP64 slices")

"""Records and values made from the staged pair lists, where words and lanes can
go wrong: one to four words per string, electrons on both sides of a word
boundary, a continuum of either spin, and lists long enough that a warp queues
single substitutions over several steps."""
import pytest

from gpu_util import assert_blocks_close, gpu_dense
from oracle import coracle
from paper_1709_03005_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


def _check(P, precision):
    o = coracle.Oracle(P)
    G, _, _ = gpu_dense(P, precision)
    assert_blocks_close(G, o.dense(), o, (1e-12, 1e-10)[precision], mixed=precision == 1)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kw", [dict(n_to=8, n_elec=5, n_words=1), dict(n_to=8, n_elec=5, n_words=4, cont_spin=1),
                                dict(n_to=66, n_elec=6, n_words=2), dict(n_to=68, n_elec=69, n_words=3, cont_spin=1)])
def test_words_and_spins(precision, kw):
    P = synth.make_tiny(9, n_co=3, n_det=40, n_groups=2, n_state=[2, 3], cont_ranges=[(0, 3), (1, 2)], n_l2=60, **kw)
    _check(P, precision)


@pytest.mark.parametrize("precision", [0, 1])
def test_long_lists(precision):
    _check(synth.make_tiny(9, n_to=18, n_elec=6, n_co=2, n_det=2000, n_state=2, n_l2=6), precision)

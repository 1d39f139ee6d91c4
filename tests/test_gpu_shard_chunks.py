"""The gamma items of a shard in the sort chunks of the whole list: 6320 single
excitations over 3200 keys take 13 chunks of 512, and the 3556 of the first of two
ranks would have taken 14 of 256."""
import numpy as np
import pytest

from gpu_util import assert_blocks_close
from oracle import coracle
from paper_1709_03005_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1709_03005_gb300 import build_ext
    build_ext.build()


def _problem():
    """Two electrons in 40 orbitals: a 15 x 15 grid of determinants (28 single
    excitations each), then 30 with next to none."""
    P = synth.make_tiny(406, n_to=40, n_co=3, n_elec=2, n_det=255, n_state=3, n_l2=8)
    alpha = [i for i in range(15) for _ in range(15)] + [15 + i % 25 for i in range(30)]
    beta = [j for _ in range(15) for j in range(15)] + [15 + (i % 25 + 5 * (i // 25) + 1) % 25 for i in range(30)]
    dets = np.array([[1 << a, 1 << b] for a, b in zip(alpha, beta)], dtype=np.uint64)
    assert len({tuple(d) for d in dets.tolist()}) == 255
    P.groups[0].dets = dets
    return P


def _singles(dets, rows):
    x = np.unpackbits((dets[rows, None, :] ^ dets[None, :, :]).view(np.uint8), axis=-1)
    return int((x.reshape(len(rows), len(dets), -1).sum(-1) == 2).sum())


@pytest.mark.parametrize("precision", [0, 1])
def test_uneven_halves(precision):
    import torch
    from paper_1709_03005_gb300 import hb
    P = _problem()
    half = _singles(P.groups[0].dets, range(127))
    assert 13 * 256 < half <= 5120 < _singles(P.groups[0].dets, range(255)) <= 13 * 512
    H = hb.Hamiltonian(P)
    reduced = sum(H.build_contract(precision, r, 2)[0].clone() for r in range(2))
    b = H.allocate()
    for r in range(2):
        H.build_expand(precision, r, 2, reduced, b)
    torch.cuda.synchronize()
    o = coracle.Oracle(P)
    assert_blocks_close(hb.dense_from_blocks(b).cpu().numpy(), o.dense(), o, 1e-10 if precision else 1e-12, "halves",
                        mixed=precision == 1)
    H.close()

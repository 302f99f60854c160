"""Delivery tiles of batch members: two blocks of the batch kernel fit an SM at every
column size, and members equal their standalone nets on both sides of the sizes
where the tile changes."""
import numpy as np
import pytest

from paper_1511_09325_gb300 import build as B
from paper_1511_09325_gb300 import snn
from paper_1511_09325_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SM_SHARED = 228 * 1024     # bytes of shared memory of an SM
PER_BLOCK = 1024 + 4336    # kept by the system, and the batch kernel's static part
LISTS = 16 * 332 * 4       # sector lists of a block's 16 warps


@pytest.fixture(scope="module", autouse=True)
def _lib():
    B.build()
    snn.load()


@pytest.mark.parametrize("npc", [1240, 1344, 1345, 1364, 1365, 2048])
def test_two_blocks_per_sm_and_same_results(npc):
    n, s = W.neuron_params(n_per_col=npc, n_exc=npc * 4 // 5), W.synapse_params(k_out=40, d_max=3)
    with snn.Batch([(4, 4), (2, 1)], [n, n], [s, s], [5, 6], "f16w") as b:
        cols = b.members[0].info()["tile"] ** 2  # the tiles of a square grid are square
        tile = cols * (-(-npc // 4) * 16 + 256) + LISTS
        assert 2 * (tile + PER_BLOCK) <= SM_SHARED
        b.step(30)
        got = [(m.spikes(), m.state()) for m in b.members]
    for (gw, gh), seed, ((st, ids, over), state) in zip([(4, 4), (2, 1)], [5, 6], got):
        with snn.Net(gw, gh, n, s, seed, "f16w") as net:
            net.step(30)
            t, i, o = net.spikes()
            assert not over and not o and len(i)
            key = lambda a, c: np.sort(np.asarray(a, np.int64) << 32 | np.asarray(c, np.int64))
            assert np.array_equal(key(st, ids), key(t, i))
            assert all(np.array_equal(x, y) for x, y in zip(state, net.state()))

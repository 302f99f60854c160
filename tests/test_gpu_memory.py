"""Nets that fit the device only with the smaller spike lists (rows in place of
descriptors) and the longest row's table stride: the same synapses, rasters and
states as with room for the descriptors, for every form that lists spikes.

The device is filled so that the last net of a form finds too little room.
"""
import contextlib

import numpy as np
import pytest
import torch

from paper_1511_09325_gb300 import build as B
from paper_1511_09325_gb300 import snn
from paper_1511_09325_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GRID, SEED, STEPS, MB = (12, 12), 21, 60, 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _lib():
    B.build()
    snn.load()


@contextlib.contextmanager
def room(left):
    """All but `left` bytes of the device taken."""
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    assert free > left
    blob = torch.empty(free - left, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del blob
        torch.cuda.empty_cache()


def _sorted(st, ids):
    return np.sort(np.asarray(st, np.int64) << 32 | np.asarray(ids, np.int64))


def _net(prec, **law):
    with snn.Net(*GRID, W.neuron_params(), W.synapse_params(**law), SEED, prec) as net:
        net.step(STEPS)
        st, ids, over = net.spikes()
        assert not over and len(ids)
        return [net.info()], [_sorted(st, ids), *net.state(), *net.synapses(1000, 8)]


def _shards(prec):
    n, s = W.neuron_params(), W.synapse_params()
    shards = [snn.Shard(*GRID, t, n, s, SEED, prec) for t in snn.split_grid(*GRID, 2, 1)]
    try:
        out = []
        for _ in range(STEPS):
            for sh in shards:
                sh.update()
            sent = np.sort(np.concatenate([sh.spikes()[1] for sh in shards]))
            out.append(sent)
            for sh in shards:
                sh.deliver(sent)
        for sh in shards:
            out += sh.state()
        return [snn.snn_info(sh.handle) for sh in shards], out
    finally:
        for sh in shards:
            sh.close()


def _batch(prec):
    n, s = W.neuron_params(), W.synapse_params()
    with snn.Batch([GRID, GRID], [n, n], [s, s], [SEED, SEED + 1], prec) as b:
        b.step(STEPS)
        out = []
        for m in b.members:
            st, ids, over = m.spikes()
            assert not over and len(ids)
            out += [_sorted(st, ids), *m.state()]
        return [m.info() for m in b.members], out


# form, its precision, MB short of room for descriptors, nets that go without.
# A net of 178 560 neurons saves 1302 B a neuron (232 MB) by its lists and
# 32 to 45 slots of each row (23 to 65 MB); the batch short of 330 MB has no room
# for its second member until the first one is built without descriptors too.
FORMS = {
    "fixed_f32w": (_net, ("f32w",), {}, 0, 1),
    "fixed_f16w": (_net, ("f16w",), {}, 0, 1),
    "paper_f16w": (_net, ("f16w",), dict(connectivity=1), 0, 1),
    "shards_f32w": (_shards, ("f32w",), {}, 100, 1),
    "batch_one_f16w": (_batch, ("f16w",), {}, 100, 1),
    "batch_one_f32w": (_batch, ("f32w",), {}, 100, 1),
    "batch_both_f16w": (_batch, ("f16w",), {}, 330, 2),
}


@pytest.mark.parametrize("name", sorted(FORMS))
def test_same_results_without_room_for_descriptors(name):
    form, args, kw, short, lean = FORMS[name]
    info0, want = form(*args, **kw)
    total = sum(i["device_bytes"] for i in info0)
    with room(total - short * MB):
        info1, got = form(*args, **kw)
    smaller = [b["device_bytes"] < a["device_bytes"] - 200 * MB for a, b in zip(info0, info1)]
    assert sum(smaller) == lean
    assert len(got) == len(want)
    for g, w in zip(got, want):
        assert np.array_equal(g, w)


@pytest.mark.parametrize("records", [1, 2000, 1 << 14, 1 << 20])
def test_synapse_readback_in_the_drain_stage(records):
    # 4 x 3 columns of 50 neurons, rows of 60: the stage holds no row, 16
    # (a buffer of its own is taken below 32), 135, or all 600
    n, s = W.neuron_params(n_per_col=50, n_exc=40), W.synapse_params(k_out=60)
    with snn.Net(4, 3, n, s, SEED, "f32w") as net:
        want = net.synapses(0, net.n)
        net.set_record_capacity(records)
        for got, w in zip(net.synapses(0, net.n), want):
            assert np.array_equal(got, w)
        net.step(5)
        assert net.synapses(0, 1)[0].shape == (1, 60)

"""A net takes the larger spike lists only where that leaves room for what fits the
device beside it without them: a second net, a pair of shards, a differentiable
view.  And a net of very small columns, whose counters weigh as much as its
neurons, builds where only the smaller lists fit.
"""
import contextlib

import numpy as np
import pytest
import torch

from paper_1511_09325_gb300 import build as B
from paper_1511_09325_gb300 import snn
from paper_1511_09325_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GRID, SEED, STEPS, MB = (12, 12), 23, 40, 1 << 20
THETA = np.array([1.0, 1.0, 1.0, 1.0, 0.02, 2.5])


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


def _build(prec, shards, seed=SEED):
    n, s = W.neuron_params(), W.synapse_params()
    if not shards:
        return snn.Net(*GRID, n, s, seed, prec)
    return snn.Shard(*GRID, snn.split_grid(*GRID, 2, 1)[seed - SEED], n, s, SEED, prec)


def _bytes(net):
    return snn.snn_info(net.handle)["device_bytes"]


def _sizes(prec, shards):
    """Device bytes of a net with descriptor lists and with lists of rows."""
    with contextlib.closing(_build(prec, shards)) as net:
        large = _bytes(net)
    with room(large), contextlib.closing(_build(prec, shards)) as net:
        return large, _bytes(net)


@pytest.mark.parametrize("shards", [False, True])
@pytest.mark.parametrize("prec", ["f32w", "f16w"])
def test_second_net_fits(prec, shards):
    large, small = _sizes(prec, shards)
    assert large > small + 200 * MB
    with room(large + small - 100 * MB):
        with contextlib.closing(_build(prec, shards)) as a, contextlib.closing(_build(prec, shards, SEED + 1)) as b:
            assert _bytes(a) == small
            if not shards:
                a.step(STEPS)
                b.step(STEPS)
                got = a.state() + b.state()
    if not shards:
        with _build(prec, False) as a, _build(prec, False, SEED + 1) as b:
            assert _bytes(a) == large
            a.step(STEPS)
            b.step(STEPS)
            assert all(np.array_equal(x, y) for x, y in zip(got, a.state() + b.state()))


def test_differentiable_view_fits():
    large, _ = _sizes("f32w", False)
    with _build("f32w", False) as net:
        free = torch.cuda.mem_get_info()[0]
        with snn.Grad(net, 30, checkpoint_every=15) as g:
            view = free - torch.cuda.mem_get_info()[0]
            want = g.loss_and_grad(THETA)
    assert view > 150 * MB
    with room(large + view - 100 * MB):
        with _build("f32w", False) as net, snn.Grad(net, 30, checkpoint_every=15) as g:
            got = g.loss_and_grad(THETA)
    assert got[0] == want[0] and np.array_equal(got[2], want[2])


def test_small_columns_where_only_the_smaller_lists_fit():
    # 4 M columns of 2: counters and list lengths of 130 MB beside the neurons
    n = W.neuron_params(n_per_col=2, n_exc=1, nu_ext_kHz=4.0)
    s = W.synapse_params(k_out=2, d_max=32)
    with snn.Net(2000, 2000, n, s, SEED, "f16w") as net:
        large = _bytes(net)
        net.step(4)
        want = net.state()
    with room(large - 30 * MB):
        with snn.Net(2000, 2000, n, s, SEED, "f16w") as net:
            assert _bytes(net) < large
            net.step(4)
            got = net.state()
    assert all(np.array_equal(x, y) for x, y in zip(got, want))

"""Table strides and spike lists.

A net takes the larger spike lists only where that leaves room for what fits the
device beside it without them: a second net, a pair of shards, a differentiable
view.  And a net of very small columns, whose counters weigh as much as its
neurons, builds where only the smaller lists fit.

The rows' stride is an estimate of the longest row; where a row is longer, the
longest one's length.
"""
import contextlib

import numpy as np
import pytest
import torch

import oracle
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


@pytest.mark.parametrize("prec", ["f32w", "f16w"])
def test_rows_longer_than_estimated(prec):
    # 20 synapses over 40 bucket parts of equal weight (all remote, a flat stencil, half
    # of it in the own 6 x 6 tile): the estimate is 152 slots, a row whose synapses all
    # lie in parts of their own takes 160
    oracle.build()
    n = W.neuron_params(n_per_col=200, n_exc=160, nu_ext_kHz=3.0)
    s = W.synapse_params(k_out=20, frac_local=0.0, lambda_cols=1e6)
    p = oracle.make_params(*GRID, n, s, SEED)
    with snn.Net(*GRID, n, s, SEED, prec) as net:
        assert net.info()["row_capacity"] == 160
        for j0 in (0, 12345, net.n - 200):
            got = net.synapses(j0, 200)
            o = oracle.synapses(p, prec, j0, 200)
            by_delay = np.argsort(o["delay"], axis=1, kind="stable")
            for g, k in zip(got, ("target", "delay", "wfx")):
                assert np.array_equal(g, np.take_along_axis(o[k], by_delay, 1))
        net.step(STEPS)
        st, ids, over = net.spikes()
        v = net.state()[0]
    o = oracle.run(p, prec, STEPS)
    key = lambda t, i: np.sort(np.asarray(t, np.int64) << 32 | np.asarray(i, np.int64))
    assert not over and len(ids) > 0
    assert np.array_equal(key(st, ids), key(o["t"], o["i"])) and np.array_equal(v.astype(np.float64), o["v"])

"""FP16 weights on both sides of 64 mV, where the delivery's conversion to input
units changes: rows, raster and state against the CPU oracle, for a net of its own
and for batch members (of which one wide net changes all members' kernel)."""
import numpy as np
import pytest

import oracle
from paper_1511_09325_gb300 import build as B
from paper_1511_09325_gb300 import snn
from paper_1511_09325_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STEPS, SEED = 60, 31
NEURON = dict(n_per_col=40, n_exc=32, nu_ext_kHz=3.0)
# excitatory and inhibitory mean and spread; 9 x 8 columns are several delivery tiles
WEIGHTS = {
    "below": (63.96875, -63.96875, 0.0),
    "at_64_exc": (64.0, -1.6, 0.0),
    "at_64_inh": (0.4, -64.0, 0.0),
    "across": (60.0, -70.0, 0.25),
    "large": (700.0, -2500.0, 0.1),
}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    B.build()
    snn.load()
    oracle.build()


def _params(name):
    e, i, cv = WEIGHTS[name]
    return W.neuron_params(**NEURON), W.synapse_params(k_out=24, w_exc_mV=e, w_inh_mV=i, w_cv=cv)


def _check(net, name, gw, gh, seed):
    n, s = _params(name)
    p = oracle.make_params(gw, gh, n, s, seed)
    st, ids, over = net.spikes()
    v, c, r = net.state()
    o = oracle.run(p, "f16w", STEPS)
    key = lambda t, i: np.sort(np.asarray(t, np.int64) << 32 | np.asarray(i, np.int64))
    assert not over and len(o["t"]) > 0
    assert np.array_equal(key(st, ids), key(o["t"], o["i"]))
    assert np.array_equal(v.astype(np.float64), o["v"])
    assert np.array_equal(c.astype(np.float64), o["c"]) and np.array_equal(r, o["r"])


@pytest.mark.parametrize("name", sorted(WEIGHTS))
def test_net_matches_oracle(name):
    n, s = _params(name)
    with snn.Net(9, 8, n, s, SEED, "f16w") as net:
        _, _, wfx = net.synapses(0, 64)
        o = oracle.synapses(oracle.make_params(9, 8, n, s, SEED), "f16w", 0, 64)
        by_delay = np.argsort(o["delay"], axis=1, kind="stable")
        assert np.array_equal(wfx, np.take_along_axis(o["wfx"], by_delay, 1))
        net.step(STEPS)
        _check(net, name, 9, 8, SEED)


def test_batch_members_match_oracle():
    names = ["below", "across", "large"]
    params = [_params(k) for k in names]
    grids = [(9, 8), (2, 2), (4, 3)]
    with snn.Batch(grids, [n for n, _ in params], [s for _, s in params], [SEED + k for k in range(3)],
                   "f16w") as b:
        b.step(STEPS)
        for k, m in enumerate(b.members):
            _check(m, names[k], *grids[k], SEED + k)

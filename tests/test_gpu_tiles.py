"""Delivery tiles, table layout and update paths at the sizes where they change,
against the CPU oracle: rows (read back in the order in which they were drawn),
raster and final state are compared exactly.

The cases are the edges of the layout: more tiles than a warp has lanes (the
block-wide range search), columns of 2, 3 and 5 neurons and of the largest size,
rows too long for units of 8 slots (units of 16), a tile that covers the whole
grid (no synapse leaves it), one bucket, descriptors of one and of six planes,
and both sides of the window threshold (quiet and saturated nets).
"""
import numpy as np
import pytest

import oracle
from paper_1511_09325_gb300 import build as B
from paper_1511_09325_gb300 import snn
from paper_1511_09325_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    B.build()
    snn.load()
    oracle.build()


def _npc(k, **kw):
    return dict(n_per_col=k, n_exc=max(1, 4 * k // 5), **kw)


CASES = {
    # 8 x 7 = 56 delivery tiles
    "56_tiles_f32w": (60, 50, _npc(8, nu_ext_kHz=3.0), dict(k_out=40), 3, "f32w", 60),
    "56_tiles_f16w": (60, 50, _npc(8, nu_ext_kHz=3.0), dict(k_out=40, d_max=3), 3, "f16w", 60),
    "columns_of_2": (9, 5, _npc(2, nu_ext_kHz=4.0), dict(k_out=12, d_min=2, d_max=5), 5, "f32w", 200),
    "columns_of_3": (7, 4, _npc(3, nu_ext_kHz=4.0), dict(k_out=12, d_max=6), 6, "f16w", 200),
    "columns_of_5": (11, 3, _npc(5, nu_ext_kHz=4.0), dict(k_out=30), 7, "f32w", 200),
    "columns_of_2048": (4, 3, _npc(2048), dict(k_out=64, d_max=4), 8, "f16w", 40),
    # K + 7 * 64 slots exceed 255 units of 8
    "units_of_16_f32w": (3, 2, _npc(101, nu_ext_kHz=3.0), dict(k_out=1750, d_max=32), 9, "f32w", 80),
    "units_of_16_f16w": (9, 2, _npc(101, nu_ext_kHz=3.0), dict(k_out=1750, d_max=32), 9, "f16w", 80),
    "one_tile": (2, 2, _npc(500, nu_ext_kHz=3.0), dict(k_out=500), 10, "f16w", 150),
    "one_bucket": (8, 3, _npc(60, nu_ext_kHz=3.0), dict(k_out=80, d_min=1, d_max=1), 11, "f32w", 150),
    "six_planes": (8, 3, _npc(60, nu_ext_kHz=3.0), dict(k_out=80, d_max=32), 12, "f16w", 150),
    "quiet": (13, 7, _npc(100, nu_ext_kHz=1.2), dict(k_out=150), 13, "f16w", 150),
    "saturated_f16w": (13, 7, _npc(100, nu_ext_kHz=20.0), dict(k_out=150), 13, "f16w", 40),
    "saturated_f32w": (13, 7, _npc(102, nu_ext_kHz=20.0), dict(k_out=150), 14, "f32w", 40),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_matches_oracle(name):
    gw, gh, nov, sov, seed, prec, steps = CASES[name]
    n, s = W.neuron_params(**nov), W.synapse_params(**sov)
    p = oracle.make_params(gw, gh, n, s, seed)
    with snn.Net(gw, gh, n, s, seed, prec) as net:
        N = net.n
        for j0 in sorted({0, N // 2, max(0, N - 40)}):
            rows = min(40, N - j0)
            tg, dl, wf = net.synapses(j0, rows)
            o = oracle.synapses(p, prec, j0, rows)
            by_delay = np.argsort(o["delay"], axis=1, kind="stable")
            for got, want in ((tg, o["target"]), (dl, o["delay"]), (wf, o["wfx"])):
                assert np.array_equal(got, np.take_along_axis(want, by_delay, 1))
        net.step(steps)
        st, ids, over = net.spikes()
        v, c, r = net.state()
        rec, _, _ = net.stats()
    o = oracle.run(p, prec, steps)
    key = lambda t, i: np.sort(np.asarray(t, np.int64) * (1 << 32) + np.asarray(i, np.int64))
    assert not over and len(o["t"]) > 0
    assert np.array_equal(key(st, ids), key(o["t"], o["i"]))
    assert np.array_equal(v.astype(np.float64), o["v"])
    assert np.array_equal(c.astype(np.float64), o["c"])
    assert np.array_equal(r, o["r"])
    assert rec == len(o["t"]) * s["k_out"]


def test_large_state_readback_and_a_second_smaller_net():
    """State arrays above the direct-copy size (staged in pieces), read twice;
    a net with a smaller window built in between leaves the first one running."""
    n, s = W.neuron_params(n_per_col=1024, n_exc=819), W.synapse_params(k_out=20, d_max=2)
    with snn.Net(33, 21, n, s, 4, "f16w") as net:
        net.step(5)
        with snn.Net(1, 1, n, s, 4, "f16w") as small:
            small.step(70)
            assert small.stats()[2] == 70
        net.step(70)
        a, b = net.state(), net.state()
        t, i, over = net.spikes()
        assert not over
    assert all(np.array_equal(x, y) for x, y in zip(a, b))
    last = i[t == 74]
    assert len(last) > 0 and np.all(a[2][last] == 2) and int((a[2] == 2).sum()) == len(last)

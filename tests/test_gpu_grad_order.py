"""The order of the FP32 sums of the surrogate gradient is part of its result: the
recorded gradients (tests/golden/grad_draw_order.json), which were summed in the
order in which a row's synapses are drawn, come out again to the rounding of the
FP64 sums over the neurons, whatever order the table keeps the synapses in.

Hundreds of steps amplify any other order of the FP32 sums: adding each bucket by
eight lanes moved these gradients by 2e-9 to 2e-6 of their largest component.
"""
import json
import os

import numpy as np
import pytest

from paper_1511_09325_gb300 import build as B
from paper_1511_09325_gb300 import snn
from paper_1511_09325_gb300 import workloads as W

pytestmark = pytest.mark.gpu

THETA = np.array([1.0, 1.0, 1.0, 1.0, 0.02, 2.5])
GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "grad_draw_order.json")


def _npc(k, e=None, **kw):
    return dict(n_per_col=k, n_exc=max(1, 4 * k // 5) if e is None else e, **kw)


# grid, neurons, synapses, seed, steps, checkpoint interval, hard spikes: tables of
# one tile and of several, units of 8 and of 16 slots, both laws, one population
CASES = {
    "cols4x4_hard": (4, 4, {}, {}, 11, 500, 50, True),
    "cols2x2_soft": (2, 2, {}, {}, 5, 8, 50, False),
    "tiles_9x8": (9, 8, _npc(200, nu_ext_kHz=3.0), dict(k_out=300), 3, 60, 25, True),
    "tiles_9x8_soft": (9, 8, _npc(200, nu_ext_kHz=3.0), dict(k_out=300), 3, 6, 50, False),
    "tiles_paper_law": (11, 8, _npc(300, nu_ext_kHz=3.0), dict(connectivity=1), 4, 50, 50, True),
    "tiles_ragged": (13, 7, _npc(1001), dict(k_out=997, stencil_radius=2, d_min=2, d_max=9), 6, 60, 20, True),
    "units_of_16": (3, 2, _npc(101, nu_ext_kHz=3.0), dict(k_out=1750, d_max=32), 9, 80, 30, True),
    "units_of_16_tiles": (20, 2, _npc(101, nu_ext_kHz=3.0), dict(k_out=1750, d_max=32), 9, 60, 30, True),
    "columns_of_2048": (2, 2, _npc(2048), dict(k_out=200, d_max=32), 8, 80, 40, True),
    "columns_of_3": (30, 4, _npc(3, nu_ext_kHz=4.0), dict(k_out=12, d_max=6), 6, 100, 40, True),
    "one_bucket": (12, 9, _npc(60, nu_ext_kHz=3.0), dict(k_out=2000, d_min=3, d_max=3), 11, 60, 60, True),
    "one_population": (3, 3, _npc(100, 100, nu_ext_kHz=3.0), dict(k_out=90), 12, 50, 50, True),
}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    B.build()
    snn.load()


@pytest.mark.parametrize("name", sorted(CASES))
def test_gradient_in_draw_order(name):
    gw, gh, nov, sov, seed, T, every, hard = CASES[name]
    with open(GOLDEN) as f:
        want = json.load(f)["cases"][name]
    n, s = W.neuron_params(**nov), W.synapse_params(**sov)
    with snn.Net(gw, gh, n, s, seed, "f32w") as net, snn.Grad(net, T, checkpoint_every=every, hard=hard) as g:
        loss, rates, grad = g.loss_and_grad(THETA)
    assert loss == want["loss"] and list(rates) == want["rates"]
    # FP64 sums of up to 9e4 partials of mixed sign in another order
    grad, ref = np.array(grad), np.array(want["grad"])
    assert np.all(np.abs(grad - ref) <= 2e-10 * np.abs(ref).max())

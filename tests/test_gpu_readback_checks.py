"""snn_read_synapses reports a row whose stored bucket ends, records or padding are
not what the seed draws: any flipped byte of a descriptor, a synapse turned into
padding, padding turned into a synapse.  Undoing the flip makes the rows readable
again, with the same contents."""
import numpy as np
import pytest

from paper_1511_09325_gb300 import build as B
from paper_1511_09325_gb300 import snn
from paper_1511_09325_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NEURON = 1234  # of 9 x 9 columns of 50: several delivery tiles


@pytest.fixture(scope="module", autouse=True)
def _lib():
    B.build()
    snn.load()


def _net(prec, law, **kw):
    n = W.neuron_params(n_per_col=50, n_exc=40)
    return snn.Net(9, 9, n, W.synapse_params(connectivity=law, **kw), 3, prec)


def _flipped(net, neuron, byte, mask, in_table):
    snn.snn_debug_flip_byte(net.handle, neuron, byte, mask, in_table)
    try:
        with pytest.raises(snn.SnnError) as e:
            net.synapses(neuron - 3, 6)
        assert e.value.code == snn.SNN_ESTATE
        net.synapses(0, neuron)  # the rows before are intact
    finally:
        snn.snn_debug_flip_byte(net.handle, neuron, byte, mask, in_table)


@pytest.mark.parametrize("law", [0, 1])
@pytest.mark.parametrize("prec", ["f32w", "f16w"])
def test_descriptor(prec, law):
    with _net(prec, law, k_out=80, d_max=8) as net:
        want = net.synapses(NEURON - 3, 6)
        # planes of 16 bytes: row (2 bytes), start, unused, then the ends of the
        # in and out parts of six buckets
        used = [0, 1, 2, *range(4, 16), 16, 17, 18, *range(20, 24)]
        for byte in used:
            _flipped(net, NEURON, byte, 1, False)
        for got, w in zip(net.synapses(NEURON - 3, 6), want):
            assert np.array_equal(got, w)


@pytest.mark.parametrize("prec", ["f32w", "f16w"])
@pytest.mark.parametrize("out", [False, True])
def test_record_and_padding(prec, out):
    # one bucket of 20 synapses to the own tile (one column: none leaves it) ...
    if not out:
        n = W.neuron_params(n_per_col=50, n_exc=40)
        net = snn.Net(1, 1, n, W.synapse_params(k_out=20, d_max=1), 3, prec)
        first, pad, neuron = 0, 21, 7
    else:
        # ... or all to other columns, some of them in other tiles
        net = _net(prec, 0, k_out=20, d_max=1, frac_local=0.0)
        neuron, first, pad = None, None, None
        npc, geo = 50, net.info()["tile"]  # 5 x 5 columns
        for j in range(7, net.n - 7, 7):  # a row with an out part that ends in padding
            t = net.synapses(j, 1)[0] // npc
            c = j // npc
            tile = lambda a: (a % 9 // geo, a // 9 // geo)
            n_in = int(sum(tile(int(a)) == tile(c) for a in t.ravel()))
            n_out = 20 - n_in
            if n_out and n_out % 8:
                first, neuron = -(-n_in // 8) * 8, j
                pad = first + n_out
                break
        assert neuron is not None
    size = 8 if prec == "f32w" else 4
    with net:
        want = net.synapses(0, net.n)
        if prec == "f32w":  # bit 31 of the code marks padding
            _flipped(net, neuron, first * size + 3, 0x80, True)
            _flipped(net, neuron, pad * size + 3, 0x80, True)
        elif out:  # stencil field dx + 3 = 7 marks padding: bits 11 .. 13
            _flipped(net, neuron, pad * size + 1, 0x08, True)
        else:  # the half 2^-24 marks padding: bits 16 .. 30
            _flipped(net, neuron, pad * size + 2, 0x02, True)
        for got, w in zip(net.synapses(0, net.n), want):
            assert np.array_equal(got, w)


def test_bad_arguments():
    with _net("f32w", 0, k_out=20) as net:
        for neuron, byte, table in ((-1, 0, 0), (net.n, 0, 0), (0, -1, 1), (0, 64, 0), (0, 1 << 20, 1)):
            with pytest.raises(snn.SnnError) as e:
                snn.snn_debug_flip_byte(net.handle, neuron, byte, 1, table)
            assert e.value.code == snn.SNN_EINVAL

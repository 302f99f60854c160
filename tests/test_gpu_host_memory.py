"""Host allocations that fail inside the library come back as SNN_ENOMEM, and the
net goes on: no C++ exception crosses the ABI.  The calls run in a process of their
own whose address space is limited around them."""
import os
import subprocess
import sys

import pytest

from paper_1511_09325_gb300 import build as B

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import contextlib, ctypes, resource
import numpy as np
from paper_1511_09325_gb300 import snn, workloads as W
L = snn.load()

@contextlib.contextmanager
def no_room():
    used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
    old = resource.getrlimit(resource.RLIMIT_AS)
    resource.setrlimit(resource.RLIMIT_AS, (used + (4 << 20), old[1]))
    try:
        yield
    finally:
        resource.setrlimit(resource.RLIMIT_AS, old)

# 4 M columns: 64 MB of counts for the rates, 32 MB of row lengths
n = W.neuron_params(n_per_col=2, n_exc=1, nu_ext_kHz=4.0)
s = W.synapse_params(k_out=2, d_max=2)
with snn.Net(2000, 2000, n, s, 1, "f16w") as net:
    net.step(3)
    rates = net.rates()
    net.step(3)
    net.stats()
    hz, pop = np.zeros(2 * net.n_cols, np.float32), np.zeros(2, np.float32)
    rows = [np.zeros(2 * net.n, t) for t in (np.int64, np.int32, np.int32)]
    ptr = [ctypes.c_void_p(a.ctypes.data) for a in (hz, pop, *rows)]
    ms = (ctypes.c_double * 2)()
    with no_room():
        rc = [L.snn_read_rates(net.handle, ptr[0], hz.size, ptr[1]),
              L.snn_read_synapses(net.handle, 0, net.n, *ptr[2:]),
              L.snn_step_profiled(net.handle, 1 << 24, ms, None),
              L.snn_step_profiled(net.handle, 1 << 60, ms, None)]
    assert rc == [snn.SNN_ENOMEM] * 4, rc
    assert snn.snn_last_error(net.handle)
    assert net.stats()[2] == 6
    net.step(1)
    assert net.rates()[0].max() > 0
    assert len(net.synapses(0, net.n)[0].ravel()) == 2 * net.n
print("done")
"""


def test_host_allocation_failures_are_reported():
    B.build()
    env = dict(os.environ, PYTHONPATH=ROOT)
    p = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, env=env, cwd=ROOT, timeout=300)
    assert p.returncode == 0 and p.stdout.strip() == "done", (p.returncode, p.stderr[-2000:])

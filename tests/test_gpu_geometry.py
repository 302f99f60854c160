"""The geometry tables of a net take no host memory per column: 4 M columns of two
neurons (256 bytes of table a column on the device) grow the process by less than
a tenth of the table."""
import os
import subprocess
import sys

import pytest

from paper_1511_09325_gb300 import build as B

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import resource
from paper_1511_09325_gb300 import snn, workloads as W
snn.load()
n = W.neuron_params(n_per_col=2, n_exc=1, nu_ext_kHz=4.0)
s = W.synapse_params(k_out=2, d_max=2)
peak = lambda: resource.getrusage(resource.RUSAGE_SELF).ru_maxrss
with snn.Net(20, 20, n, s, 1, "f16w") as net:
    net.step(2)
    net.stats()
    before = peak()
with snn.Net(2000, 2000, n, s, 1, "f16w") as net:
    grown = peak() - before
    net.step(2)
    assert net.stats()[2] == 2
print("grown", grown)
"""


def test_no_host_memory_per_column():
    B.build()
    env = dict(os.environ, PYTHONPATH=ROOT)
    p = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, env=env, cwd=ROOT, timeout=300)
    assert p.returncode == 0, p.stderr
    assert int(p.stdout.split()[-1]) * 1024 < 4_000_000 * 256 // 10

"""Device memory that a layer's phases take beyond the tables (needs a GB300).

In a process of its own each, whose memory pool starts empty: what the pool maps
shows in the device's free memory and stays mapped until the process ends."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

pytestmark = pytest.mark.gpu

GROWTH = """
import torch
import paper_2512_12094_gb300 as pp
import pp_inputs as pi
torch.empty(1, device="cuda")
wl = pi.config0_heisenberg(%d, 0.05, 3)
p = pp.Propagator.from_workload(wl, symmetry=0)
before = torch.cuda.mem_get_info()[0]
for layer in reversed(range(3)):
    gx, gz, th = wl.circuit.gate_arrays(layer)
    p.apply_layer(gx, gz, th, True)
print(before - torch.cuda.mem_get_info()[0], p.stats()["device_bytes"])
"""


def taken(script):
    out = subprocess.run([sys.executable, "-c", script], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    return [int(v) for v in out.stdout.split()]


@pytest.mark.parametrize("n", [3, 5, 8])
def test_buckets_are_not_sized_beyond_the_strings_there_are(n):
    """The first layer multiplies its one term by thousands; the layers after it
    cannot hold more than 4^n strings.  The bound: 1824 buckets (12 warps on 152
    SMs) of at most 256 + 4 * 368 records of 32 bytes, twice, is 0.2 GB, and a
    bucket for every 368 strings beyond as many buckets adds none at these n."""
    import paper_2512_12094_gb300 as pp
    pp.build()
    used, tables = taken(GROWTH % n)
    assert used <= tables + (512 << 20)


DESTROY = """
import numpy as np, torch
import paper_2512_12094_gb300 as pp
torch.empty(1, device="cuda")
rng = np.random.default_rng(0)
m = 30000000
x, z = (rng.integers(0, 1 << 32, (m, 1), dtype=np.uint64) for _ in range(2))
c = rng.random(m)
before = torch.cuda.mem_get_info()[0]
p = pp.Propagator(32, x, z, c, symmetry=0)
during = torch.cuda.mem_get_info()[0]
p.close()
print(before - during, before - torch.cuda.mem_get_info()[0])
"""


def test_memory_of_a_large_context_goes_back():
    """Two tables of 120 million strings and their indexes are over 10 GB; 8 GiB of it
    may stay mapped for the next context."""
    import paper_2512_12094_gb300 as pp
    pp.build()
    during, after = taken(DESTROY)
    assert during > 9 << 30
    assert after <= (8 << 30) + (64 << 20)

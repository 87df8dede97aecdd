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


LARGE = """
import sys
import numpy as np, torch
import paper_2512_12094_gb300 as pp
torch.empty(1, device="cuda")
rng = np.random.default_rng(0)
m, n = 30000000, 32
x, z = (rng.integers(0, 1 << n, (m, 1), dtype=np.uint64) for _ in range(2))
before = torch.cuda.mem_get_info()[0]
p = pp.Propagator(n, x, z, np.full(m, 1e-3), symmetry=0, eps=5e-4)
tables = before - torch.cuda.mem_get_info()[0]
gx = np.array([[1 << q] for q in range(8)], dtype=np.uint64)
p.apply_layer(gx, np.zeros_like(gx), np.full(8, 0.05), True)  # births of 5e-5 are truncated
routes = pp.pp_debug_layer_routes(p.ctx)
during = before - torch.cuda.mem_get_info()[0]
p.close()
print(tables, during, before - torch.cuda.mem_get_info()[0], routes["phased"])
"""


def test_scratch_of_a_large_layer_goes_back():
    """45 million strings expected are 64 thousand buckets of 3056 records of 32 bytes,
    twice: 12 GB beside the tables, of which 8 GiB may stay for the next context."""
    import paper_2512_12094_gb300 as pp
    pp.build()
    tables, during, after, phased = taken(LARGE)
    assert phased == 1 and during > tables + (11 << 30)
    assert after <= during - (12 << 30) + (8 << 30) + (64 << 20)

"""pp_set_grid_fraction and the wait limits of neighbours where layers are phased (needs
a GB300)."""
import numpy as np
import pytest

import paper_2512_12094_gb300 as pp
import pp_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    pp.build()
    pp.load()


def sorted_table(prop):
    x, z, c = prop.export()
    order = np.lexsort((*x.T, *z.T))
    return x[order], z[order], c[order]


def run(wl, fraction, symmetry=0):
    """(table, device ms of the last layer's gates, routes)"""
    p = pp.Propagator.from_workload(wl, symmetry=symmetry, profile=True)
    pp.pp_set_grid_fraction(p.ctx, fraction)
    for layer in reversed(range(len(wl.circuit.layers))):
        before = p.stats()["gate_kernel_ms"]
        gx, gz, th = wl.circuit.gate_arrays(layer)
        p.apply_layer(gx, gz, th, True)
    ms = p.stats()["gate_kernel_ms"] - before
    out = sorted_table(p), ms, pp.pp_debug_layer_routes(p.ctx)
    p.close()
    return out


def test_phases_keep_to_the_fraction():
    """A table of hundreds of thousands of strings, whose phases fill the chip: on a
    sixteenth of it the last layer takes several times as long, and the table is the
    same bit for bit."""
    wl = pi.config1_ring(n=32, steps=11, eps=2e-5, max_weight=10)
    (a, ms_a, ra), (b, ms_b, rb) = run(wl, 1.0), run(wl, 1.0 / 16)
    assert ra["phased"] == rb["phased"] == 11 and len(a[2]) > 200000
    for u, v in zip(a, b):
        np.testing.assert_array_equal(u, v)
    assert ms_b > 3.0 * ms_a


@pytest.mark.parametrize("fraction", [1e-6, 0.01, 0.37])
def test_small_fractions(fraction):
    wl = pi.config1_ring(n=20, steps=4, eps=1e-4, max_weight=8)
    (a, _, _), (b, _, _) = run(wl, 1.0), run(wl, fraction)
    for u, v in zip(a, b):
        np.testing.assert_array_equal(u, v)


@pytest.mark.parametrize("B,f32,fraction", [(40, False, 0.01), (300, True, 0.3)])
def test_rows_on_a_fraction(B, f32, fraction):
    n = 20
    angles = pi.batched_ring_angles(B, 1)
    gx, gz, _ = pi.Circuit(n, [pi.ring_layer(n, 0.0, 0.0, 0.0)]).gate_arrays(0)
    x, z, c = pi.mean_z(n).arrays()
    tables = []
    for f in (1.0, fraction):
        p = pp.Propagator(n, x, z, np.repeat(c[:, None], B, axis=1), eps=1e-5, batch=B, f32=f32)
        pp.pp_set_grid_fraction(p.ctx, f)
        for _ in range(3):
            p.apply_layer(gx, gz, np.repeat(angles.T, n, axis=0), True)
        tables.append(sorted_table(p))
        p.close()
    for u, v in zip(*tables):
        np.testing.assert_array_equal(u, v)


def test_served_jobs_with_a_wait_limit_among_phased_ones():
    """A wait limit of 50 ms, which a barrier's wait is far below on the job's own share
    of the GPU."""
    jobs, want = [], []
    for k in range(12):
        limit = 50000 if k % 3 == 0 else 0
        n, steps, eps = (24, 8, 1e-5) if limit else (32, 9, 3e-5)
        wl = pi.config1_ring(n=n, steps=steps, eps=eps, max_weight=8, symmetry=1)
        cfg = pp.pp_config_default(n_qubits=n, symmetry=1, coeff_eps=eps, max_weight=8, wait_limit=limit)
        x, z, c = wl.observable.arrays()
        gx, gz, th = wl.circuit.gate_arrays(0)
        jobs.append(pp.make_job(cfg, x, z, c, pp.pack_gates(gx, gz), th, steps, wl.state.bloch, True, 0))
        want.append((n, wl))
    values = {}
    for n, wl in want:
        if n not in values:
            p = pp.Propagator.from_workload(wl, symmetry=1)
            values[n] = p.run(wl)
            p.close()
    server = pp.pp_server_create(4, 16 << 30, 0)
    res = [pp.pp_server_wait(server, i) for i in [pp.pp_submit(server, j) for j, _ in jobs]]
    pp.pp_server_destroy(server)
    for r, (n, _) in zip(res, want):
        assert r["status"] == 0, r["message"]
        assert r["value"] == pytest.approx(values[n], abs=1e-10)

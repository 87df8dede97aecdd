"""Wait limits beside contexts whose phases take the whole GPU (needs a GB300)."""
import threading

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


def apply_all(prop, wl):
    for layer in reversed(range(len(wl.circuit.layers))):
        gx, gz, th = wl.circuit.gate_arrays(layer)
        prop.apply_layer(gx, gz, th, True)


@pytest.mark.parametrize("batch", [1, 40])
def test_a_short_wait_limit_beside_phases(batch):
    """A context with a wait limit of 20 ms on a quarter of the GPU, beside two that
    keep all of it busy with phases: its blocks start apart, which its limit does not
    count, and it gives what it gives alone."""
    n = 40 if batch == 1 else 20
    wl = pi.config1_ring(n=n, steps=5, eps=1e-4, max_weight=7)
    gx, gz, th = wl.circuit.gate_arrays(0)
    x, z, c = wl.observable.arrays()
    if batch > 1:
        c, th = np.repeat(c[:, None], batch, axis=1), np.repeat(th[:, None], batch, axis=1)

    def job():
        p = pp.Propagator(n, x, z, c, eps=1e-4, max_weight=7, batch=batch, wait_limit=20000)
        pp.pp_set_grid_fraction(p.ctx, 0.25)
        for _ in range(5):
            p.apply_layer(gx, gz, th, True)
        t = sorted_table(p)
        assert not any(pp.pp_debug_layer_routes(p.ctx).values())
        p.close()
        return t

    want = job()
    stop, errors = threading.Event(), []

    def neighbour():
        busy = pi.config1_ring(n=32, steps=11, eps=1e-5, max_weight=10)
        try:
            while not stop.is_set():
                p = pp.Propagator.from_workload(busy, symmetry=0)
                apply_all(p, busy)
                p.close()
        except Exception as e:  # shown below
            errors.append(e)

    side = [threading.Thread(target=neighbour) for _ in range(2)]
    for t in side:
        t.start()
    try:
        for _ in range(8):
            for u, v in zip(job(), want):
                np.testing.assert_array_equal(u, v)
    finally:
        stop.set()
        for t in side:
            t.join()
    assert not errors, errors


def test_served_jobs_with_a_wait_limit_among_phased_ones():
    """A wait limit of 50 ms, which a barrier's wait is far below once all blocks run."""
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

"""Persistent launches resumed after a stall while other contexts keep the GPU full, so
that their blocks do not start together (needs a GB300)."""
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


def table_of(prop):
    x, z, c = prop.export()
    order = np.lexsort((*x.T, *z.T))
    return x[order], z[order], c[order]


def apply_all(prop, wl):
    for layer in reversed(range(len(wl.circuit.layers))):
        gx, gz, th = wl.circuit.gate_arrays(layer)
        prop.apply_layer(gx, gz, th, True)


@pytest.mark.parametrize("n", [40, 64])
def test_resumed_layers_beside_phases(n):
    """Almost no headroom, so that layers stop for room at gate after gate (also at
    those whose number is one above a multiple of three, which resume in the slot
    their own births are counted in); a phased job runs beside them throughout."""
    wl = pi.config1_ring(n=n, steps=6, eps=3e-5, max_weight=7)
    kw = dict(symmetry=0, block_threads=256, room_factor=0.01)
    alone = pp.Propagator.from_workload(wl, **kw)
    apply_all(alone, wl)
    want, stats = table_of(alone), alone.stats()
    alone.close()
    assert stats["stalls"] > 3
    stop, errors = threading.Event(), []

    def neighbour():
        busy = pi.config1_ring(n=32, steps=10, eps=2e-5, max_weight=10)
        try:
            while not stop.is_set():
                p = pp.Propagator.from_workload(busy, symmetry=0)
                apply_all(p, busy)
                p.close()
        except Exception as e:  # shown below
            errors.append(e)

    def job():
        try:
            for _ in range(12):
                p = pp.Propagator.from_workload(wl, **kw)
                pp.pp_set_grid_fraction(p.ctx, 0.25)
                apply_all(p, wl)
                for u, v in zip(table_of(p), want):
                    np.testing.assert_array_equal(u, v)
                assert p.stats()["gate_updates"] == stats["gate_updates"]
                p.close()
        except Exception as e:
            errors.append(e)

    side = threading.Thread(target=neighbour)
    side.start()
    jobs = [threading.Thread(target=job) for _ in range(3)]
    for t in jobs:
        t.start()
    for t in jobs:
        t.join()
    stop.set()
    side.join()
    assert not errors, errors

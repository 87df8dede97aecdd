"""Which way a layer went: as phases, given up and applied by the persistent
kernel, merged by buckets or by the index (pp_debug_layer_routes).  Every way gives
the same table, so a comparison of tables does not show that one was taken (needs a
GB300)."""
import numpy as np
import pytest

import paper_2512_12094_gb300 as pp
import pp_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    pp.build()
    pp.load()


def routes_of(wl, symmetry, **kw):
    """(routes, entries of the table)"""
    p = pp.Propagator.from_workload(wl, symmetry=symmetry, **kw)
    for layer in reversed(range(len(wl.circuit.layers))):
        gx, gz, th = wl.circuit.gate_arrays(layer)
        p.apply_layer(gx, gz, th, True)
    r, n = pp.pp_debug_layer_routes(p.ctx), p.num_terms()[0]
    p.close()
    return r, n


GIVEN_UP = ("bucket_full", "class_full", "table_full")


@pytest.mark.parametrize("n,eps,wmax", [(32, 1e-4, 10), (64, 1e-4, 8), (40, 0.0, 4), (100, 1e-3, 6)])
def test_ring_layers_are_phased(n, eps, wmax):
    """Dense phases of one and two words, sparse ones with and without truncation."""
    r, _ = routes_of(pi.config1_ring(n=n, steps=6, eps=eps, max_weight=wmax), 0)
    assert r["phased"] == 6 and not any(r[k] for k in GIVEN_UP)


@pytest.mark.parametrize("kw", [dict(block_threads=256), dict(wait_limit=10 ** 7), dict(layer_kernel=False),
                                dict(budget=4 << 20)])
def test_layers_that_are_not(kw):
    """The settings that name the other kernels, and a budget without room for the
    buckets: 304 buckets of 256 records of 32 bytes, twice, take 5 MB."""
    wl = pi.config1_ring(n=32, steps=4, eps=1e-3, max_weight=10)
    r, _ = routes_of(wl, 0, **kw)
    assert not any(r.values())


@pytest.mark.parametrize("group,n,by_buckets,least", [(1, 32, True, 6), (3, 24, True, 6), (2, 24, False, 1)])
def test_merges_of_phased_layers(group, n, by_buckets, least):
    if group == 2:
        wl = pi.config2_all_to_all(n, 0.02, 3, 0.01, 1e-4, 1, 2)
    else:
        wl = pi.config1_ring(n=n, steps=11, eps=1e-4, max_weight=9)
    r, _ = routes_of(wl, group)
    assert r["phased"] >= least
    assert (r["merge_buckets"] > 0) == by_buckets and r["merge_full"] == 0


@pytest.mark.parametrize("B,f32", [(64, False), (100, True)])
def test_batched_layers_are_phased(B, f32):
    n = 24
    angles = pi.batched_ring_angles(B, 1)
    gx, gz, _ = pi.Circuit(n, [pi.ring_layer(n, 0.0, 0.0, 0.0)]).gate_arrays(0)
    x, z, c = pi.mean_z(n).arrays()
    p = pp.Propagator(n, x, z, np.repeat(c[:, None], B, axis=1), eps=1e-5, batch=B, f32=f32)
    for _ in range(2):
        p.apply_layer(gx, gz, np.repeat(angles.T, n, axis=0), True)
    assert pp.pp_debug_layer_routes(p.ctx)["phased"] == 2
    p.close()


def test_a_full_table_is_counted():
    r, _ = routes_of(pi.config1_ring(n=40, steps=5, eps=1e-5, max_weight=7), 0, room_factor=0.01)
    assert r["table_full"] > 0


@pytest.mark.parametrize("n,eps,steps,last", [(9, 0.0, 3, False), (10, 0.0, 3, False), (10, 1e-6, 4, False),
                                              (14, 2e-4, 3, True), (20, 1e-3, 3, True)])
def test_full_tables_of_wide_classes_are_not_phased(n, eps, steps, last):
    """All-to-all layers, whose phases are not dense, on tables that hold a large
    share of the 4^n strings: the last layer is the persistent kernel's, at once and
    not after a phase was given up; on more qubits it stays phased."""
    wl = pi.config0_heisenberg(n, 0.05, steps)
    wl.eps = eps
    p = pp.Propagator.from_workload(wl, symmetry=0)
    for layer in reversed(range(steps)):
        before = pp.pp_debug_layer_routes(p.ctx)
        gx, gz, th = wl.circuit.gate_arrays(layer)
        p.apply_layer(gx, gz, th, True)
    after = pp.pp_debug_layer_routes(p.ctx)
    p.close()
    assert after["phased"] - before["phased"] == int(last)
    assert all(after[k] == before[k] for k in GIVEN_UP)


@pytest.mark.parametrize("n", [8, 10])
def test_full_tables_of_dense_phases_are(n):
    r, entries = routes_of(pi.config1_ring(n=n, steps=8, eps=1e-6, max_weight=-1), 0)
    assert entries > 4 ** n // 4 and r["phased"] == 8


@pytest.mark.parametrize("lx,ly,steps", [(5, 5, 7), (6, 6, 6)])
def test_classes_outgrow_their_room_once_of_a_kind(lx, ly, steps):
    """Bonds of every site without a weight limit: a layer of a large table is given
    up for a class of more than ten active gates, or of more strings than a warp holds;
    the layers after it are cut so that no class can be, and are phased again."""
    wl = pi.torus_ising(lx, ly, steps, 0.4, 0.6, 0.3, 2e-4, -1, pp.sym_torus(lx))
    p = pp.Propagator.from_workload(wl, symmetry=wl.symmetry)
    b = pp.Propagator.from_workload(wl, symmetry=wl.symmetry, block_threads=256)
    seen = []
    for layer in reversed(range(steps)):
        gx, gz, th = wl.circuit.gate_arrays(layer)
        p.apply_layer(gx, gz, th, True)
        b.apply_layer(gx, gz, th, True)
        assert p.num_terms()[0] == b.num_terms()[0]
        seen.append(pp.pp_debug_layer_routes(p.ctx))
    p.close()
    b.close()
    assert 1 <= seen[-1]["class_full"] <= 3
    assert seen[-1]["phased"] == seen[-2]["phased"] + 1 or seen[-1]["class_full"] == seen[-2]["class_full"] + 1
    assert sum(r["class_full"] == 1 for r in seen) > 1  # it is not every layer's lot


def test_a_layer_that_grew_is_phased_again():
    """Half of the strings, letters I and Z drawn evenly, hold a letter that a rotation
    of one site turns.  Four such rotations, one that does not commute with them, and
    four more multiply the strings 25 times in the first layer; the second, whose table
    is full in these sites, is phased too."""
    n, terms = 24, 8192
    rng = np.random.default_rng(1)
    z = np.unique(rng.integers(0, 1 << n, 2 * terms, dtype=np.uint64))[:terms]
    p = pp.Propagator(n, np.zeros_like(z)[:, None], z[:, None], rng.uniform(0.5, 1.0, len(z)), symmetry=0,
                      eps=1e-6, room_factor=10.0)
    gates = [("x", q) for q in range(4)] + [("z", 0)] + [("x", q) for q in range(4, 8)]
    gx = np.array([[1 << q if k == "x" else 0] for k, q in gates], dtype=np.uint64)
    gz = np.array([[1 << q if k == "z" else 0] for k, q in gates], dtype=np.uint64)
    th = np.full(len(gates), 0.3)
    for _ in range(2):
        p.apply_layer(gx[::-1].copy(), gz[::-1].copy(), th, True)
    r, grown = pp.pp_debug_layer_routes(p.ctx), p.num_terms()[0]
    p.close()
    assert grown > 10 * terms
    assert r["phased"] == 2


def test_tuning_leaves_the_plan_as_it_was():
    """Tuned before a layer whose phases are given up (a class is too large): the trials
    are not counted, and the layers after it are given up no more often, and phased no
    less often if phases were chosen, than in a context that was not tuned."""
    wl = pi.torus_ising(5, 6, 6, 0.4, 0.6, 0.3, 1e-4, -1, pp.sym_torus(5))
    tuned = pp.Propagator.from_workload(wl, symmetry=wl.symmetry)
    plain = pp.Propagator.from_workload(wl, symmetry=wl.symmetry)
    for k, layer in enumerate(reversed(range(6))):
        gx, gz, th = wl.circuit.gate_arrays(layer)
        g = pp.pack_gates(gx, gz)
        if k in (2, 4):
            before = pp.pp_debug_layer_routes(tuned.ctx)
            pp.pp_tune(tuned.ctx, g, th)
            assert pp.pp_debug_layer_routes(tuned.ctx) == before
        pp.pp_apply_layer(tuned.ctx, g, th, True)
        pp.pp_apply_layer(plain.ctx, g, th, True)
        assert tuned.num_terms()[0] == plain.num_terms()[0]
    a, b = pp.pp_debug_layer_routes(tuned.ctx), pp.pp_debug_layer_routes(plain.ctx)
    assert b["class_full"] >= 1
    for k in GIVEN_UP:
        assert a[k] <= b[k]
    tuned.close()
    plain.close()

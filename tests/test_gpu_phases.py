"""Layers applied as phases over bucketed strings against the persistent layer
kernel (block_threads=256 asks for it) and the per-gate path's oracle: the same
strings, coefficients bit for bit and update statistics, at every word count,
with and without truncation, noise and groups, on runs of gates that commute
and runs that do not, on tables of one string and of millions (needs a GB300)."""
import numpy as np
import pytest

import oracle
import paper_2512_12094_gb300 as pp
import pp_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    pp.build()
    pp.load()
    oracle.build()


def sorted_table(prop):
    x, z, c = prop.export()
    order = np.lexsort((*x.T, *z.T))
    return x[order], z[order], c[order]


KEYS = ("gate_updates", "anticommuting_terms", "gates_applied", "live_terms")


def run_pair(wl, symmetry, exact=True):
    a = pp.Propagator.from_workload(wl, symmetry=symmetry)
    b = pp.Propagator.from_workload(wl, symmetry=symmetry, block_threads=256)
    for layer in reversed(range(len(wl.circuit.layers))):
        gx, gz, th = wl.circuit.gate_arrays(layer)
        a.apply_layer(gx, gz, th, True)
        b.apply_layer(gx, gz, th, True)
        if exact:
            assert a.num_terms()[0] == b.num_terms()[0]
    sa, sb = a.stats(), b.stats()
    ta, tb = sorted_table(a), sorted_table(b)
    for k in KEYS:
        assert sa[k] == sb[k], k
    np.testing.assert_array_equal(ta[0], tb[0])
    np.testing.assert_array_equal(ta[1], tb[1])
    if exact:
        np.testing.assert_array_equal(ta[2], tb[2])
    else:  # merges sum with atomics: each layer's sums round in any order
        np.testing.assert_allclose(ta[2], tb[2], rtol=0, atol=1e-12)
    a.close()
    b.close()
    return sa, len(ta[2])


@pytest.mark.parametrize("n,layers,eps,wmax", [
    (1, 2, 0.0, -1), (2, 3, 0.0, -1), (3, 3, 0.0, -1), (9, 4, 0.0, -1), (16, 4, 0.0, 5),
    (32, 9, 1e-4, 10), (33, 4, 1e-3, -1), (63, 4, 1e-4, 8), (64, 4, 1e-4, 8), (65, 4, 1e-4, 8),
    (127, 4, 0.0, 3), (150, 4, 1e-3, 6), (200, 3, 1e-4, 7)])
def test_ring_bit_for_bit(n, layers, eps, wmax):
    wl = pi.config1_ring(n=n, steps=layers, eps=eps, max_weight=wmax)
    run_pair(wl, 0)


@pytest.mark.parametrize("group,n,layers,eps,wmax", [
    (1, 17, 6, 1e-4, 8), (3, 12, 5, 1e-4, -1), (1, 70, 5, 1e-4, 6), (1, 32, 11, 1e-4, 10)])
def test_merged_rings(group, n, layers, eps, wmax):
    wl = pi.config1_ring(n=n, steps=layers, eps=eps, max_weight=wmax)
    run_pair(wl, group, exact=False)


def test_large_table_with_wide_classes():
    """Two bonds of every site on a torus without a weight limit: hundreds of
    thousands of strings, classes of hundreds, buckets done in parts and layers
    given up and applied by the persistent kernel."""
    wl = pi.torus_ising(5, 6, 4, eps=1e-4)
    _, n_plain = run_pair(wl, 0)
    assert n_plain > 100000
    _, n_merged = run_pair(wl, pp.sym_torus(5), exact=False)
    assert n_merged > 100000


@pytest.mark.parametrize("noise_mode", [1, 2])
def test_noise(noise_mode):
    wl = pi.config1_ring(n=20, steps=5, eps=1e-5, max_weight=7)
    wl.noise_mode, wl.noise_p = noise_mode, 0.02
    run_pair(wl, 0)


@pytest.mark.parametrize("n,gates,support,terms,eps", [
    (6, 40, 3, 20, 0.0), (12, 30, 2, 50, 1e-3), (40, 60, 3, 200, 0.1), (130, 60, 1, 300, 0.0),
    (255, 40, 2, 100, 1e-2)])
def test_random_circuits(n, gates, support, terms, eps):
    circ = pi.random_circuit(n, 3, gates, seed=n, max_support=support)
    obs = pi.random_observable(n, terms, seed=n + 1, max_weight=4)
    wl = pi.Workload("r", circ, obs, pi.zero_state(n), eps=eps, max_weight=-1)
    run_pair(wl, 0)


def test_all_to_all_sublayers_against_the_oracle():
    wl = pi.xxz_all_to_all(10, 0.05, 3, eps=1e-5, symmetry=2, split=True)
    prop = pp.Propagator.from_workload(wl, symmetry=2)
    ox, oz, oc = wl.observable.arrays()
    st = oracle.OracleState(10, ox, oz, oc, group=2, eps=wl.eps, max_weight=-1)
    for layer in reversed(range(len(wl.circuit.layers))):
        gx, gz, th = wl.circuit.gate_arrays(layer)
        prop.apply_layer(gx, gz, th)
        st.apply_layer(gx, gz, th, group=2)
    assert prop.stats()["gate_updates"] == st.updates
    assert prop.num_terms()[0] == len(st)
    assert prop.expect(wl.state.bloch) == pytest.approx(st.expect(wl.state.bloch, 2), abs=1e-12)
    prop.close()


def test_table_grows_past_its_room_and_back_to_gates():
    """With almost no headroom the destination fills up: the layer is given
    up, applied by the persistent kernel (which grows the table), and the
    result is the same."""
    wl = pi.config1_ring(n=40, steps=5, eps=1e-5, max_weight=7)
    a = pp.Propagator.from_workload(wl, symmetry=0, room_factor=0.01)
    b = pp.Propagator.from_workload(wl, symmetry=0, block_threads=256)
    a.run(wl)
    b.run(wl)
    ta, tb = sorted_table(a), sorted_table(b)
    for u, v in zip(ta, tb):
        np.testing.assert_array_equal(u, v)
    assert a.stats()["gate_updates"] == b.stats()["gate_updates"]
    a.close()
    b.close()


def test_phases_with_a_memory_budget():
    """A budget without room for the buckets keeps the other path, with room
    for them it does not; the tables agree."""
    wl = pi.config1_ring(n=24, steps=5, eps=1e-5, max_weight=7)
    tables = []
    for budget in (0, 64 << 20, 2 << 30):
        p = pp.Propagator.from_workload(wl, symmetry=0, budget=budget)
        p.run(wl)
        tables.append(sorted_table(p))
        p.close()
    for t in tables[1:]:
        for u, v in zip(tables[0], t):
            np.testing.assert_array_equal(u, v)


def batched_pair(n, B, f32, eps, wmax, layers, group=0):
    angles = pi.batched_ring_angles(B, n)
    gx, gz, _ = pi.Circuit(n, [pi.ring_layer(n, 0.0, 0.0, 0.0)]).gate_arrays(0)
    th = np.repeat(angles.T, n, axis=0)
    th = th[:, 0].copy() if B == 1 else th
    x, z, c = pi.mean_z(n).arrays()
    coef = np.repeat(c[:, None], B, axis=1)
    kw = dict(symmetry=group, eps=eps, max_weight=wmax, batch=B, f32=f32)
    a = pp.Propagator(n, x, z, coef, **kw)
    b = pp.Propagator(n, x, z, coef, block_threads=256, **kw)
    for _ in range(layers):
        a.apply_layer(gx, gz, th, True)
        b.apply_layer(gx, gz, th, True)
        assert a.num_terms()[0] == b.num_terms()[0]
    sa, sb = a.stats(), b.stats()
    for k in KEYS:
        assert sa[k] == sb[k], k
    ta, tb = sorted_table(a), sorted_table(b)
    np.testing.assert_array_equal(ta[0], tb[0])
    np.testing.assert_array_equal(ta[1], tb[1])
    if group == 0:
        np.testing.assert_array_equal(ta[2], tb[2])
    else:
        np.testing.assert_allclose(ta[2], tb[2], rtol=0, atol=1e-6 if f32 else 1e-12)
    a.close()
    b.close()
    return len(ta[0])


@pytest.mark.parametrize("n,B,f32,eps,wmax,layers", [
    (1, 4, False, 0.0, -1, 2), (5, 3, False, 0.0, -1, 3), (9, 1, True, 1e-4, -1, 4),
    (16, 31, True, 1e-4, 6, 3), (32, 33, False, 1e-5, -1, 3), (33, 256, False, 1e-5, -1, 2),
    (64, 256, True, 1e-5, -1, 3), (40, 300, False, 1e-4, 5, 2), (12, 512, False, 1e-6, -1, 3),
    (11, 64, False, 0.0, -1, 4)])
def test_rows_bit_for_bit(n, B, f32, eps, wmax, layers):
    """Rows at column counts below, at and above a block, both types, classes
    that fit shared memory and classes that do not."""
    batched_pair(n, B, f32, eps, wmax, layers)


@pytest.mark.parametrize("f32", [False, True])
def test_rows_merged(f32):
    assert batched_pair(14, 20, f32, 1e-4, -1, 3, group=1) > 100

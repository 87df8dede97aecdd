"""Merge by buckets in shared memory against the hash-index merge of the oracle:
the same representatives and sums, for every group it takes and every key width,
at list lengths on both sides of its rules, with strings that are all distinct, in
full orbits, or all one (where it gives up for the index), and inside layers
(needs a GB300)."""
import numpy as np
import pytest

import oracle
import paper_2512_12094_gb300 as pp
import pp_inputs as pi

pytestmark = pytest.mark.gpu

EDGE = 65536


@pytest.fixture(scope="module", autouse=True)
def _built():
    pp.build()
    pp.load()
    oracle.build()


def merged_on_gpu(n, code, x, z, c):
    import torch
    W = (n + 63) // 64
    keys = torch.from_numpy(np.concatenate([x, z], axis=1).view(np.int64)).cuda()
    coef = torch.from_numpy(c).cuda()
    out_k, out_c = torch.empty_like(keys), torch.empty_like(coef)
    m = pp.pp_merge_terms(n, code, len(c), keys, coef, out_k, out_c)
    k = out_k[:m].cpu().numpy().view(np.uint64)
    return k[:, :W], k[:, W:], out_c[:m].cpu().numpy()


def merged_on_host(n, code, x, z, c):
    cx, cz = oracle.canonical(n, code, x, z)
    rows = np.concatenate([cx, cz], axis=1)
    order = np.lexsort(rows.T)
    rows, vals = rows[order], c[order]
    first = np.r_[True, (rows[1:] != rows[:-1]).any(axis=1)]
    seg = np.cumsum(first) - 1
    sums = np.zeros(seg[-1] + 1)
    np.add.at(sums, seg, vals)
    mags = np.zeros(seg[-1] + 1)
    np.add.at(mags, seg, np.abs(vals))
    return rows[first], sums, mags, np.bincount(seg)


def random_strings(rng, n, m, distinct):
    """Strings of a few sites drawn from ``distinct`` ones."""
    W = (n + 63) // 64
    base = np.zeros((distinct, 2 * W), dtype=np.uint64)
    for _ in range(min(n, 7)):
        site = rng.integers(0, n, distinct)
        letter = rng.integers(1, 4, distinct)
        bit = np.uint64(1) << (site % 64).astype(np.uint64)
        rows = np.arange(distinct)
        base[rows, site // 64] ^= bit * (letter & 1).astype(np.uint64)
        base[rows, W + site // 64] ^= bit * (letter >> 1).astype(np.uint64)
    pick = base[rng.integers(0, distinct, m)]
    return np.ascontiguousarray(pick[:, :W]), np.ascontiguousarray(pick[:, W:])


@pytest.mark.parametrize("n,code,m,distinct", [
    (17, 0, 1, 1), (17, 1, 2, 1), (40, 1, 255, 100), (100, 3, 1000, 1), (8, 1, EDGE - 1, 40000),
    (8, 0, EDGE, 40000), (8, 1, EDGE + 1, 40000), (17, 1, EDGE + 1, 40000),
    (32, 1, 300007, 300000), (32, 3, 200001, 5000), (30, pp.sym_torus(5), 150001, 150000),
    (64, 1, EDGE, EDGE), (65, 1, 100003, 60000), (128, 3, 80001, 80000), (130, 0, 90001, 30000),
    (192, 1, 70001, 70000), (256, 1, 70001, 40000), (9, 1, 500009, 400), (20, 1, 1 << 17, 1)])
def test_merge_list(n, code, m, distinct):
    rng = np.random.default_rng(100 + n)
    x, z = random_strings(rng, n, m, distinct)
    c = rng.standard_normal(m)
    gx, gz, gc = merged_on_gpu(n, code, x, z, c)
    rows, sums, mags, size = merged_on_host(n, code, x, z, c)
    got = np.concatenate([gx, gz], axis=1)
    order = np.lexsort(got.T)
    np.testing.assert_array_equal(got[order], rows)
    # each side's sum of k terms is within k ulp of the sum of magnitudes
    bound = 2 * size * np.finfo(float).eps * mags
    assert (np.abs(gc[order] - sums) <= bound).all()


def test_special_values_and_zero_sums():
    n, m = 20, EDGE + 5
    rng = np.random.default_rng(5)
    x, z = random_strings(rng, n, m, m // 2)
    c = np.where(rng.random(m) < 0.5, 0.0, -0.0)
    c[:3] = [np.inf, -np.inf, np.nan]
    gx, gz, gc = merged_on_gpu(n, 1, x, z, c)
    rows, sums, _, _ = merged_on_host(n, 1, x, z, c)
    got = np.concatenate([gx, gz], axis=1)
    order = np.lexsort(got.T)
    np.testing.assert_array_equal(got[order], rows)  # zero sums stay entries
    np.testing.assert_array_equal(gc[order], sums)


@pytest.mark.parametrize("group,n,steps,eps", [(1, 32, 12, 1e-4), (3, 24, 10, 1e-4), (1, 70, 8, 1e-4)])
def test_layers_merge_by_buckets(group, n, steps, eps):
    """Merged layers of tens of thousands of strings, against the persistent
    kernel's with the merge by the index; sums of at most 2 n terms of magnitude
    at most one a layer."""
    wl = pi.config1_ring(n=n, steps=steps, eps=eps, max_weight=9)
    a = pp.Propagator.from_workload(wl, symmetry=group)
    b = pp.Propagator.from_workload(wl, symmetry=group, block_threads=256)
    most = 0
    for layer in reversed(range(len(wl.circuit.layers))):
        gx, gz, th = wl.circuit.gate_arrays(layer)
        a.apply_layer(gx, gz, th, True)
        b.apply_layer(gx, gz, th, True)
        most = max(most, a.num_terms()[0])
    assert most >= 1024
    ta, tb = a.export(), b.export()
    oa, ob = np.lexsort((*ta[0].T, *ta[1].T)), np.lexsort((*tb[0].T, *tb[1].T))
    np.testing.assert_array_equal(ta[0][oa], tb[0][ob])
    np.testing.assert_array_equal(ta[1][oa], tb[1][ob])
    np.testing.assert_allclose(ta[2][oa], tb[2][ob], rtol=0, atol=1e-12)
    a.close()
    b.close()

"""The Z_n orbit average in a product state by windows of four sites against the
oracle's, on lists on both sides of the rule that chooses it, at the smallest and
largest site counts it takes and those whose windows run over the ends of the
ring and of a word (needs a GB300)."""
import numpy as np
import pytest

import oracle
import paper_2512_12094_gb300 as pp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    pp.build()
    pp.load()
    oracle.build()


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 31, 32, 33, 63, 64, 65, 67, 101, 104, 105, 128])
@pytest.mark.parametrize("extra", [-1, 0, 1027])
def test_average_by_windows(n, extra):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m = sms * 2048 + extra
    rng = np.random.default_rng(1000 * n + extra + 1)
    distinct, W = 501, (n + 63) // 64
    letters = rng.integers(0, 4, (distinct, n)) * (rng.random((distinct, n)) < rng.random((distinct, 1)))
    x = np.zeros((distinct, W), dtype=np.uint64)
    z = np.zeros((distinct, W), dtype=np.uint64)
    for q in range(n):
        x[:, q // 64] |= (letters[:, q] & 1).astype(np.uint64) << np.uint64(q % 64)
        z[:, q // 64] |= (letters[:, q] >> 1).astype(np.uint64) << np.uint64(q % 64)
    bloch = rng.uniform(-1.0, 1.0, (n, 3))
    ov = oracle.sym_overlap(n, 1, x, z, bloch)
    pick = np.arange(m) % distinct
    c = rng.standard_normal(m)
    c[::97] = 0.0
    keys = torch.from_numpy(np.concatenate([x, z], axis=1)[pick].view(np.int64)).cuda()
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    pp.pp_overlap_sum(n, pp.SYM_ZN, m, keys, torch.from_numpy(c).cuda(),
                      torch.from_numpy(bloch).cuda(), out)
    got = float(out.cpu()[0])
    want = float(np.dot(c, ov[pick]))
    # products of at most n factors and a mean of n of them on either side,
    # magnitudes at most one, then sums of at most a few strings a thread
    assert abs(got - want) <= 2 * (2 * n + 64) * np.finfo(float).eps * np.abs(c).sum()

"""The S_n orbit-averaged overlap table against the oracle's average, at the
sizes where its launches change shape: one site, a block of one and of several
warps of z values, one and several words (needs a GB300)."""
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


@pytest.mark.parametrize("n", [1, 2, 31, 32, 63, 65, 130])
def test_sn_overlaps_match_the_oracle(n):
    import torch
    W = (n + 63) // 64
    terms = min(4 ** n, 40)
    obs = pi.random_observable(n, terms, seed=n)
    x, z, c = obs.arrays()
    bloch = pi.random_product_state(n, n + 1).bloch
    ov = oracle.sym_overlap(n, 2, x, z, bloch)
    want = float(np.sum(c * ov))
    keys = torch.from_numpy(np.concatenate([x, z], axis=1).view(np.int64)).cuda()
    assert keys.shape[1] == 2 * W
    out = torch.empty(1, dtype=torch.float64, device="cuda")
    pp.pp_overlap_sum(n, pp.SYM_SN, terms, keys, torch.from_numpy(c).cuda(),
                      torch.from_numpy(bloch).cuda(), out)
    # every site's step is a convex combination of earlier values (at most 1 in
    # size) with at most 8 roundings
    bound = 8 * n * 2.0 ** -53 * float(np.sum(np.abs(c))) + 1e-300
    assert abs(float(out.item()) - want) <= 2 * bound

"""One group of more peaks than the nucleus loop keeps flags for in registers
(65,536), on the 16-CTA and the 8-CTA clusters and on a block: sites too far
apart to reach one another, so every site has the haloes it has as a group of its
own, which the oracle computes."""
import numpy as np
import pytest

import oracle as O
from paper_2110_11408_gb300 import cso

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
BOX = 1 << 21
U = 32768


@pytest.fixture(scope="module")
def sites():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(8)
    m = 41
    at = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3) * 1.4 + rng.uniform(-0.1, 0.1, (m ** 3, 3))
    # at 300 sites the peak has 60 particles about it, so that its radius reaches
    # the third peak there and alpha times it the second
    full = rng.choice(m ** 3, 300, replace=False)
    near = rng.normal(size=(300, 60, 3))
    near *= 0.05 * rng.random((300, 60, 1)) / np.linalg.norm(near, axis=2, keepdims=True)
    x = np.concatenate([at, at[full] + [-0.41, 0, 0], at[full] + [0, 0.59, 0], (at[full][:, None] + near).reshape(-1, 3)])
    site = np.concatenate([np.arange(m ** 3), full, full, np.repeat(full, 60)])
    T = int(max(cso.cso_params_default(U).T_min_L1, cso.cso_params_default(U).T_min_L2))
    sums = np.concatenate([3 * T + rng.permutation(m ** 3), 2 * T + np.arange(600), T + 1 + rng.permutation(18000)])
    sums[full] += 10 * T
    pos = np.mod(np.rint(x * U).astype(np.int64), BOX).astype(np.int32)
    mix = rng.permutation(len(pos))
    pos, site, sums = pos[mix], site[mix], sums[mix].astype(np.int64)
    ids = np.arange(len(pos), dtype=np.uint64)
    own = np.full(m ** 3, len(pos), np.uint64)
    np.minimum.at(own, site, ids)
    l1, l2, halos, _ = O.compaso(pos, ids, sums, own[site], O.params(U))
    assert len(np.unique(l1)) == m ** 3 + 300 and m ** 3 > 65536 and len(halos) == 300
    return pos, ids, sums, l1, l2, halos


@pytest.mark.parametrize("flags,huge", [(cso.FLAG_BATCHED, 64), (cso.FLAG_BATCHED, 1 << 30), (0, 0)])
def test_one_group_of_many_peaks(sites, flags, huge):
    pos, ids, sums, l1, l2, halos = sites
    with cso.Context(0, flags=flags) as ctx:
        if huge:
            cso.cso_set_schedule(ctx.h, 64, 64)
            cso.cso_set_huge_group(ctx.h, huge)
        g1, g2, gh = cso.cso_levels(ctx.h, pos, ids, sums, np.zeros(len(pos), np.uint64), cso.cso_params_default(U))
    assert np.array_equal(g1, l1) and np.array_equal(g2, l2)
    for f in ("nucleus_id", "N", "R2", "l2max_id", "l2max_N", "n_l2"):
        assert np.array_equal(gh[f], halos[f]), f

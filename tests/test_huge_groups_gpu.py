"""L1 and L2 of one group on the 16-CTA clusters, with dozens of nuclei of small
radii in a wide background (runs of tiles, tries held in registers), some of
them with hundreds of members at one distance, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2110_11408_gb300 import cso

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
BOX = 1 << 21
U = 32768


def one_group(n, sites, seed):
    """A background of 30 particles per u^3 and `sites` clumps in it; sums that
    peak at the clumps.  Every fourth clump has a third of its members at one
    place, a quarter of u from its centre."""
    rng = np.random.default_rng(seed)
    field = int(0.8 * n)
    side = (field / 30) ** (1 / 3)
    m = rng.multinomial(n - field, rng.dirichlet(np.full(sites, 2.0)))
    c = rng.uniform(0, side, (sites, 3))
    x = [rng.uniform(0, side, (field, 3))]
    for k in range(sites):
        r = 0.02 + (m[k] / 1500) ** (1 / 3) * rng.random(m[k])
        v = rng.normal(size=(m[k], 3))
        v /= np.linalg.norm(v, axis=1, keepdims=True)
        if k % 4 == 0:
            r[: m[k] // 3], v[: m[k] // 3] = 0.25, [1, 0, 0]
        x.append(c[k] + r[:, None] * v)
    x = np.concatenate(x)
    f = sum((1 + 0.05 * k) * np.exp(-((x - c[k]) ** 2).sum(1) / 0.3) for k in range(sites))
    pos = np.mod(np.rint((x - side / 2) * U).astype(np.int64), BOX).astype(np.int32)
    sigma = (cso.cso_params_default(U).T_L0 * (2 + 1000 * f)).astype(np.int64)
    return pos, rng.permutation(n).astype(np.uint64), sigma, np.zeros(n, np.uint64)


@pytest.mark.parametrize("n,sites,flags", [(9000, 6, (0, cso.FLAG_SELECT_STRESS)), (40000, 14, (0, cso.FLAG_SELECT_STRESS)),
                                           (280000, 40, (0,))])
def test_one_huge_group(n, sites, flags):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pos, ids, sigma, l0 = one_group(n, sites, n)
    o1, o2, oh, _ = O.compaso(pos, ids, sigma, l0, O.params(U))
    assert len(np.unique(o1)) > sites
    for extra in flags:
        with cso.Context(0, flags=cso.FLAG_BATCHED | extra) as ctx:
            cso.cso_set_schedule(ctx.h, 64, 64)
            cso.cso_set_huge_group(ctx.h, 64)
            l1, l2, halos = cso.cso_levels(ctx.h, pos, ids, sigma, l0, cso.cso_params_default(U))
        assert np.array_equal(l1, o1) and np.array_equal(l2, o2)
        for f in ("nucleus_id", "N", "R2", "l2max_id", "l2max_N", "n_l2"):
            assert np.array_equal(halos[f], oh[f]), f

"""L1 and L2 inside caller-given groups of particles with 64-bit ids: sums of 62
bits, and sums none of which is above the L0 threshold, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2110_11408_gb300 import cso

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
BOX = 1 << 21
U = 32768


@pytest.mark.parametrize("sums", ["wide", "low"])
def test_levels_with_wide_ids(sums):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(3)
    n, groups = 4000, 40
    g = rng.integers(0, groups, n)
    centre = np.stack([g % 4, g // 4 % 4, g // 16], 1) * 8 * U
    pos = np.mod(np.rint(centre + rng.normal(size=(n, 3)) * 0.2 * U).astype(np.int64), BOX).astype(np.int32)
    ids = rng.integers(1 << 63, (1 << 64) - 2, n, dtype=np.uint64)
    p, po = cso.cso_params_default(U), O.params(U)
    sigma, _ = O.density(pos, po)
    if sums == "wide":
        sigma = sigma * ((1 << 62) // int(sigma.max()))
    else:
        sigma = np.minimum(sigma, int(p.T_L0) - np.arange(n) % 7)
    l0 = np.array([ids[g == k].min() for k in range(groups)], np.uint64)[g]
    w1, w2, wh, _ = O.compaso(pos, ids, sigma, l0, po)
    for flags in (0, cso.FLAG_BATCHED):
        with cso.Context(0, flags=flags) as ctx:
            l1, l2, halos = cso.cso_levels(ctx.h, pos, ids, sigma, l0, p)
        assert np.array_equal(l1, w1) and np.array_equal(l2, w2)
        assert np.array_equal(halos["nucleus_id"], wh["nucleus_id"]) and np.array_equal(halos["N"], wh["N"])
    assert len(wh) == 0 if sums == "low" else len(wh) >= groups // 2

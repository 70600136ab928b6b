"""L1 and L2 inside caller-given groups whose sizes sit at the edges of the
level kernels (a warp, the 128-, 256- and 1024-thread blocks, clusters; whole
tiles and remainders), each with several density peaks, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2110_11408_gb300 import cso, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
BOX = 1 << 21
U = 32768
SIZES = [1, 2, 31, 33, 64, 65, 127, 129, 511, 512, 513, 1025, 2047, 2048, 2049, 2177, 4097, 9000]


@pytest.fixture(scope="module")
def groups():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(17)
    pos, l0, used = [], [], 0
    for k, n in enumerate(SIZES):
        # sites 12 mean spacings apart, the first on the periodic corner
        at = np.array([k % 5, k // 5 % 5, k // 25], float) * 12 * U
        nc = int(rng.integers(1, 7))
        share = rng.multinomial(n, rng.dirichlet(np.ones(nc)))
        for m in share:
            c = at + rng.uniform(-1, 1, 3) * U * min(2.5, 0.3 * n ** (1 / 3))
            r = U * float(synth.r200(max(m, 8))) * rng.random(m) ** 2
            v = rng.normal(size=(m, 3))
            pos.append(c + r[:, None] * v / np.linalg.norm(v, axis=1, keepdims=True))
        l0 += [used] * n
        used += n
    pos = np.mod(np.rint(np.concatenate(pos)).astype(np.int64), BOX).astype(np.int32)
    ids = np.arange(used, dtype=np.uint64)
    perm = rng.permutation(used)
    pos, l0 = pos[perm], np.array(l0, np.uint64)[perm]
    # a group's label is its smallest id
    for g in np.unique(l0):
        l0[l0 == g] = ids[l0 == g].min()
    po = O.params(U)
    sigma, _ = O.density(pos, po)
    l1, l2, halos, _ = O.compaso(pos, ids, sigma, l0, po)
    return pos, ids, sigma, l0, dict(l1=l1, l2=l2, halos=halos)


@pytest.mark.parametrize("flags,bins", [(0, None), (cso.FLAG_BATCHED, None), (cso.FLAG_SELECT_STRESS, None),
                                        (cso.FLAG_BATCHED | cso.FLAG_SELECT_STRESS, None),
                                        (cso.FLAG_BATCHED, (64, 32, 1 << 30)), (cso.FLAG_BATCHED, (64, 64, 64)),
                                        (cso.FLAG_BATCHED | cso.FLAG_SELECT_STRESS, (64, 64, 64)),
                                        (cso.FLAG_BATCHED | cso.FLAG_RADIAL_BINS, (1024, 64, 4096))])
def test_levels_at_the_edges_of_the_tiers(groups, flags, bins):
    pos, ids, sigma, l0, o = groups
    p = cso.cso_params_default(U)
    with cso.Context(0, flags=flags) as ctx:
        if bins:
            cso.cso_set_schedule(ctx.h, bins[0], bins[1])
            cso.cso_set_huge_group(ctx.h, bins[2])
        l1, l2, halos = cso.cso_levels(ctx.h, pos, ids, sigma, l0, p)
    assert np.array_equal(l1, o["l1"]) and np.array_equal(l2, o["l2"])
    assert len(np.unique(o["l1"])) > len(SIZES)  # several nuclei in some groups
    for f in ("nucleus_id", "N", "R2", "l2max_id", "l2max_N", "l2_top5_N", "n_l2"):
        assert np.array_equal(halos[f], o["halos"][f]), f

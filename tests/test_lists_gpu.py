"""L0 from caller-given kernel sums at the edges of the list kernels (a warp's
run, a tile, several tiles; every particle dense, every other one, one in
fifty, none), and the whole path on the same particles, against the oracle."""
import numpy as np
import pytest

import oracle as O
from parity_util import assert_matches_oracle
from paper_2110_11408_gb300 import cso

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
BOX = 1 << 21
U = 32768


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = cso.Context(0, flags=cso.FLAG_BATCHED)
    yield c
    c.close()


def clumps(n, seed):
    """Clumps of a few cells around the periodic corner and loose particles
    between them, so that cells hold from none to hundreds of particles."""
    rng = np.random.default_rng(seed)
    k = rng.integers(0, 6, n)
    centre = rng.uniform(-3, 3, (6, 3)) * U
    width = np.array([0.05, 0.2, 0.4, 0.8, 1.5, 3.0])[k] * U
    pos = centre[k] + rng.normal(size=(n, 3)) * width[:, None]
    ids = rng.permutation(n).astype(np.uint64) + np.uint64(rng.integers(0, 1 << 40))
    return np.mod(np.rint(pos).astype(np.int64), BOX).astype(np.int32), ids


@pytest.mark.parametrize("n", [1, 31, 33, 511, 513, 4095, 4096, 4097, 8193, 13000])
@pytest.mark.parametrize("dense", ["all", "half", "few", "none"])
def test_fof_from_given_sums(ctx, n, dense):
    pos, ids = clumps(n, n)
    p, po = cso.cso_params_default(U), O.params(U)
    on = {"all": np.ones(n, bool), "half": np.arange(n) % 2 == 0, "few": np.arange(n) % 50 == 7,
          "none": np.zeros(n, bool)}[dense]
    sigma = np.where(on, int(p.T_L0) + 1 + np.arange(n), int(p.T_L0)).astype(np.int64)
    want, _ = O.fof(pos, ids, sigma, po)
    assert np.array_equal(cso.cso_fof(ctx.h, pos, ids, sigma, p), want)


@pytest.mark.parametrize("n", [1, 40, 511, 513, 4096, 4097, 13000])
def test_whole_path(ctx, n):
    pos, ids = clumps(n, 100 + n)
    assert_matches_oracle(ctx.find_groups(pos, ids, cso.cso_params_default(U), halo_cap=max(16, n)), pos, ids, U)


@pytest.mark.parametrize("n", [2, 1023, 1025, 2047, 2048, 2049])
def test_levels_with_labels_about_the_one_block_sort(ctx, n):
    pos, ids = clumps(n, 200 + n)
    po = O.params(U)
    sigma, _ = O.density(pos, po)
    rng = np.random.default_rng(n)
    l0 = np.full(n, np.iinfo(np.uint64).max, np.uint64)
    which = rng.integers(0, 7, n)
    for g in range(6):  # a seventh of the particles stays in no group
        l0[which == g] = ids[which == g].min() if (which == g).any() else 0
    l1, l2, halos = cso.cso_levels(ctx.h, pos, ids, sigma, l0, cso.cso_params_default(U))
    w1, w2, wh, _ = O.compaso(pos, ids, sigma, l0, po)
    assert np.array_equal(l1, w1) and np.array_equal(l2, w2)
    assert np.array_equal(halos["nucleus_id"], wh["nucleus_id"]) and np.array_equal(halos["R2"], wh["R2"])

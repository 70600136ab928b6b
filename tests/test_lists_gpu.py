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

"""The dense cell table: sizes about the edges of its scan and of its 16-bit
counts, and cells with more particles than 16 bits hold, against the oracle."""
import numpy as np
import pytest

import oracle as O
from parity_util import assert_matches_oracle
from paper_2110_11408_gb300 import cso

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
BOX = 1 << 21


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = cso.Context(0, flags=cso.FLAG_BATCHED)
    yield c
    c.close()


def cells_per_side(u):
    return int(BOX / np.sqrt(float(cso.cso_params_default(u).b2)))


# 128 cells a side (the fewest), either side of 2^24 cells, a run of more than
# four rounds, the many cells of a large box, the most
@pytest.mark.parametrize("u,nc", [(40960, 128), (20560, 255), (20480, 256), (16000, 327), (8192, 640), (4064, 1290)])
def test_table_sizes(ctx, u, nc):
    assert cells_per_side(u) == nc
    rng = np.random.default_rng(u)
    n = 3000
    centre = np.concatenate([rng.uniform(0, BOX, (5, 3)), [[0, 0, 0], [BOX - 1] * 3]])
    pos = centre[rng.integers(0, 7, n)] + rng.normal(size=(n, 3)) * 0.3 * u
    pos = np.mod(np.rint(pos).astype(np.int64), BOX).astype(np.int32)
    ids = rng.permutation(n).astype(np.uint64)
    assert_matches_oracle(ctx.find_groups(pos, ids, cso.cso_params_default(u), halo_cap=n), pos, ids, u)


# all of a cell at one place, so that its sums follow from one pair's share
@pytest.mark.parametrize("even,odd", [(65535, 65535), (65536, 3), (65537, 3), (3, 65537), (70000, 70001)])
def test_cells_of_more_than_16_bits(ctx, even, odd):
    u = 20000
    nc = cells_per_side(u)
    assert nc ** 3 > 1 << 24
    side = BOX / nc
    place = [np.array([int((100 + k) * side + 2), int(40 * side + 5), int(60 * side + 7)], np.int32) for k in (0, 1)]
    pos = np.concatenate([np.tile(place[0], (even, 1)), np.tile(place[1], (odd, 1))])
    where = np.repeat([0, 1], [even, odd])
    mix = np.random.default_rng(even + odd).permutation(len(pos))
    po = O.params(u)
    alone = int(O.density(pos[:1], po)[0][0])
    same = int(O.density(np.stack([place[0]] * 2), po)[0][0]) - alone
    across = int(O.density(np.stack(place), po)[0][0]) - alone
    want = np.array([alone + (even - 1) * same + odd * across, alone + (odd - 1) * same + even * across])
    got = cso.cso_density(ctx.h, pos[mix], len(pos), cso.cso_params_default(u))
    assert np.array_equal(got, want[where[mix]])

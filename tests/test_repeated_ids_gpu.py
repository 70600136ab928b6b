"""Requests whose ids repeat (a caller who wants the catalogue only and passes
zeros): equal sums are then in cell order, as with ids that number the
particles in cell order, so the same haloes come out."""
import numpy as np
import pytest

from paper_2110_11408_gb300 import cso

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
BOX = 1 << 21
U = 32768


def mirrored(m, seed, at):
    """A clump of m particles and its mirror image, a little apart: every sum
    appears twice.  Two particles share the place of the clump's peak."""
    rng = np.random.default_rng(seed)
    r = U * 0.5 * (m / 300) ** (1 / 3) * rng.random(m) ** 2
    v = rng.normal(size=(m, 3))
    p = np.rint(r[:, None] * v / np.linalg.norm(v, axis=1, keepdims=True)).astype(np.int64)
    p[0] = p[1] = 0
    p[:, 0] += int(rng.uniform(0.3, 0.9) * U * (m / 300) ** (1 / 3))
    return np.concatenate([p, p * [-1, 1, 1]]) + at


def cell_order(pos, nc):
    c = pos.astype(np.int64) * nc >> 21
    return np.lexsort((np.arange(len(pos)), pos[:, 0], c[:, 0], c[:, 1], c[:, 2]))


@pytest.mark.parametrize("flags", [0, cso.FLAG_BATCHED, cso.FLAG_BATCHED | cso.FLAG_SELECT_STRESS])
def test_repeated_ids_give_the_same_haloes(flags):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sizes = [20] * 12 + [150] * 12 + [700] * 12 + [2000] * 3 + [12000] * 2
    grid = [np.array([k % 4, k // 4 % 4, k // 16]) * 14 * U + 5 * U for k in range(len(sizes))]
    pos = np.concatenate([mirrored(m, k, grid[k]) for k, m in enumerate(sizes)])
    pos = np.mod(pos, BOX).astype(np.int32)
    pos = pos[np.random.default_rng(1).permutation(len(pos))]
    p = cso.cso_params_default(U)
    ranked = np.empty(len(pos), np.uint64)
    ranked[cell_order(pos, int(BOX / np.sqrt(float(p.b2))))] = np.arange(len(pos), dtype=np.uint64)
    with cso.Context(0, flags=flags) as ctx:
        want = ctx.find_groups(pos, ranked, p)
        zeros = [ctx.find_groups(pos, np.zeros_like(ranked), p) for _ in range(3)]
    assert len(want["halos"]) > len(sizes)
    rows = lambda h: sorted(zip(h["N"], h["R2"], map(tuple, h["com"]), h["n_l2"], h["l2max_N"]))  # noqa: E731
    for got in zeros:
        assert rows(got["halos"]) == rows(want["halos"])
        assert np.array_equal(got["l1"] == cso.NO_GROUP, want["l1"] == cso.NO_GROUP)
        assert np.array_equal(got["l2"] == cso.NO_GROUP, want["l2"] == cso.NO_GROUP)

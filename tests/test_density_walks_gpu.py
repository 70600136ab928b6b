"""Kernel sums at the edges of the density pass: warps that share rows in
every arithmetic form (signed and modulo 2^32, by the cell side), wide and
narrow x spans, the lane-by-lane walk, tiles with remainders, and the
periodic corner, against a brute-force sum over all pairs in int64."""
import numpy as np
import pytest

from paper_2110_11408_gb300 import cso

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
BOX = 1 << 21


def brute(pos, b2, query):
    p = torch.from_numpy(pos.astype(np.int64)).cuda()
    out = []
    for q in p[:query].split(256):
        d = (q[:, None, :] - p[None, :, :] + BOX // 2) % BOX - BOX // 2
        out.append((b2 - (d * d).sum(-1)).clamp(min=0).sum(1) - b2)
    return torch.cat(out).cpu().numpy()


def points(u, n, shape, seed):
    rng = np.random.default_rng(seed)
    b = 0.4 * u
    if shape == "ball":  # dense core over the periodic corner, thin halo around it
        r = b * 2.5 * rng.random(n) ** 2
        v = rng.normal(size=(n, 3))
        x = r[:, None] * v / np.linalg.norm(v, axis=1, keepdims=True)
    elif shape.startswith("even"):  # the first 32 particles fill exactly so many cells of one row
        side = BOX / int(BOX / np.sqrt(float(np.rint(b * b))))
        x = np.column_stack([np.ceil(10 * side) + np.arange(n) * (int(shape[4:]) * side - 1) / 32,
                             np.full((n, 2), 10.5 * side)])
    elif shape == "rod":  # one row of cells, many columns, across the x edge
        x = np.column_stack([rng.uniform(-6 * b, 6 * b, n), rng.uniform(0, 0.9 * b, n), rng.uniform(0, 0.9 * b, n)])
    elif shape == "spot":  # every particle on one grid point or beside it
        x = rng.integers(0, 2, (n, 3)).astype(np.float64)
    else:  # sparse background patch
        x = rng.uniform(-12 * b, 12 * b, (n, 3))
    return np.mod(np.rint(x).astype(np.int64), BOX).astype(np.int32)


# cell sides around the bounds of the forms: 16,384 (largest), 13,190, 9,490
# and 9,447 (either side of the signed form's bound), 6,575 (spans of up to 4
# cells), 5,269 (6), 3,931 (8), 3,277, 1,626
@pytest.mark.parametrize("u", [40960, 32768, 23640, 23600, 16384, 13147, 9822, 8192, 4064])
@pytest.mark.parametrize("shape,n", [("ball", 3001), ("rod", 1500), ("patch", 2000), ("spot", 257), ("ball", 33),
                                     ("ball", 1), ("even5", 45), ("even7", 45), ("even9", 45)])
def test_sums_equal_brute_force(u, shape, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = cso.cso_params_default(u)
    pos = points(u, n, shape, seed=u + n)
    query = n if n < 100 else n - 7
    with cso.Context(0) as ctx:
        got = cso.cso_density(ctx.h, pos, query, p)
    assert np.array_equal(got, brute(pos, int(p.b2), query))

"""Radial statistics and shrinking spheres of haloes of every kind of kernel (a
warp, blocks of 256 and 1024 threads, clusters), against the oracle."""
import numpy as np
import pytest

import oracle as O
from parity_util import assert_matches_oracle
from paper_2110_11408_gb300 import cso, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
BOX = 1 << 21
U = 32768


@pytest.mark.parametrize("flags", [0, cso.FLAG_BATCHED])
def test_haloes_of_every_size(flags):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(5)
    sizes = [100, 900, 1100, 4600, 5600, 7000, 19000, 24000, 50000]
    pos = []
    for k, n in enumerate(sizes):  # the first on the periodic corner
        c = np.array([k % 3, k // 3, 0]) * 16.0 * U
        r = float(synth.r200(n)) * U * rng.random(n) ** 1.5
        v = rng.normal(size=(n, 3))
        pos.append(c + r[:, None] * v / np.linalg.norm(v, axis=1, keepdims=True))
    pos = np.mod(np.rint(np.concatenate(pos)).astype(np.int64), BOX).astype(np.int32)
    pos = pos[rng.permutation(len(pos))]
    ids = np.arange(len(pos), dtype=np.uint64)
    with cso.Context(0, flags=flags) as ctx:
        g = ctx.find_groups(pos, ids, cso.cso_params_default(U), radial=True)
    o = assert_matches_oracle(g, pos, ids, U)
    N = o["halos"]["N"]
    for lo, hi in ((35, 700), (700, 4096), (4096, 16384), (16384, 1 << 30)):
        assert ((N >= lo) & (N < hi)).any(), (lo, hi)
    want = O.radial(pos, o["l1"], o["halos"], U)
    for f in want.dtype.names:
        assert np.array_equal(g["radial"][f], want[f]), f
    ss = O.shrink_sphere(pos, ids, o["l1"], o["halos"])
    for f, fo in (("ss_centre", "centre"), ("ss_n", "n"), ("ss_R2", "R2"), ("ss_iter", "iter")):
        assert np.array_equal(g["radial"][f], ss[fo]), f

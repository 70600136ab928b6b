"""A slab stream whose window's cell table counts in 16 bits first (2^24 cells
and more), with a cell that holds more, against the same box at once."""
import numpy as np
import pytest

from paper_2110_11408_gb300 import cso

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
BOX = 1 << 21
U = 8192
NC = 640


@pytest.mark.parametrize("heap", [65535, 70000])
def test_window_of_many_cells(heap):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = cso.cso_params_default(U)
    assert int(BOX / np.sqrt(float(p.b2))) == NC
    rng = np.random.default_rng(heap)
    side = BOX / NC
    # columns 4 to 63, so that one slab's window alone has 60 * 640^2 cells
    loose = np.stack([rng.uniform(4 * side, 64 * side, 3000), *rng.uniform(0, BOX, (2, 3000))], 1)
    loose[:60, 0] = (np.arange(60) + 4.5) * side
    far = np.stack([rng.uniform(300 * side, 310 * side, 50), *rng.uniform(0, BOX, (2, 50))], 1)
    one = np.array([20 * side + 100, 30 * side + 100, 40 * side + 100])
    pos = np.concatenate([np.tile(one, (heap, 1)), one + rng.normal(size=(500, 3)) * 0.3 * U, loose, far])
    pos = np.rint(pos).astype(np.int32)[rng.permutation(heap + 3550)]
    ids = rng.permutation(len(pos)).astype(np.uint64)
    with cso.Context(0, flags=cso.FLAG_BATCHED) as ctx:
        whole = ctx.find_groups(pos, ids, p, halo_cap=len(pos))
    edges = [0, BOX // 4, BOX]
    with cso.Context(0, flags=cso.FLAG_BATCHED | cso.FLAG_SLOTS(1)) as ctx:
        slabs = []
        for lo, hi in zip(edges, edges[1:]):
            m = (pos[:, 0] >= lo) & (pos[:, 0] < hi)
            b = cso.Buffers(pos[m], ids[m], False, halo_cap=len(pos), x_lo=lo, x_hi=hi, request_id=3, out_device=True)
            slabs.append((m, b, ctx.submit(b, p)))
        for m, b, t in slabs:
            assert ctx.wait(t) == (True, cso.CSO_OK), cso.cso_last_error()
            r = b.result()
            for k in ("sigma", "l0", "l1", "l2"):
                assert np.array_equal(r[k], whole[k][m]), k

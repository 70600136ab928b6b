"""Device memory of a context with a budget: what its slab streams have given
back makes room for the requests that come after them."""
import numpy as np
import pytest

from paper_2110_11408_gb300 import cso

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
BOX = 1 << 21
U = 16384
N = 2_000_000
MIB = 1 << 20


def run(budget, served):
    """A box in four slabs, as three streams side by side, then whole (served, or
    by a direct call): device memory taken after each."""
    rng = np.random.default_rng(4)
    pos = rng.integers(0, BOX, (N, 3)).astype(np.int32)
    pos = torch.from_numpy(pos[np.argsort(pos[:, 0])]).cuda()
    ids = torch.arange(N, device="cuda")
    p = cso.cso_params_default(U)
    edges = [BOX * k // 4 for k in range(5)]
    cut = np.searchsorted(pos[:, 0].cpu().numpy(), edges)
    slabs = [cso.Buffers(pos[a:b].contiguous(), ids[a:b].contiguous(), True, x_lo=lo, x_hi=hi, request_id=k)
             for a, b, lo, hi in zip(cut, cut[1:], edges, edges[1:]) for k in range(3)]
    box = cso.Buffers(pos, ids, True)
    torch.cuda.synchronize()
    taken = [torch.cuda.mem_get_info()[0]]
    with cso.Context(0, budget_bytes=budget, flags=cso.FLAG_SLOTS(1)) as ctx:
        for t in [ctx.submit(b, p) for b in slabs]:
            assert ctx.wait(t) == (True, cso.CSO_OK), cso.cso_last_error()
        taken.append(torch.cuda.mem_get_info()[0])
        if served:
            assert ctx.wait(ctx.submit(box, p)) == (True, cso.CSO_OK), cso.cso_last_error()
        else:
            cso.cso_find_groups(ctx.h, box, p)
        taken.append(torch.cuda.mem_get_info()[0])
    return taken[0] - taken[1], taken[0] - taken[2]


@pytest.mark.parametrize("served", [True, False])
def test_kept_memory_makes_room(served):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nc = int(BOX / np.sqrt(float(cso.cso_params_default(U).b2)))
    workspace = 440 * N + 8 * (nc ** 3 + 1) + 64 * MIB
    budget = workspace + (N // 16 + 1024) * 2 * cso.HALO_DTYPE.itemsize  # what the whole box reserves
    run(0, served)  # (kernels are loaded at their first launch)
    after_stream, after_box = run(budget, served)
    if served:  # one slot, whose workspace the box has grown: no more than the budget in all
        assert after_box <= budget + 32 * MIB
    else:  # the stream's memory goes when the context's own workspace comes
        assert after_box - after_stream <= workspace - 32 * MIB

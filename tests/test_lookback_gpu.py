"""Look-backs (the list ranks and the one-sweep sort) that do not wait for an
earlier tile but count its elements themselves, as one does whose patience is
used up: the whole path, and the steps on caller-given labels, against the
oracle, and tiles of large arrays against a context whose look-backs wait."""
import numpy as np
import pytest

import oracle as O
from parity_util import assert_matches_oracle
from paper_2110_11408_gb300 import cso, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def impatient():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return cso.Context(0, flags=cso.FLAG_BATCHED | cso.FLAG_SELECT_STRESS)


def test_whole_path_and_steps():
    pos, ids, meta = synth.tiny(seed=91)
    u = meta["u"]
    p, po = cso.cso_params_default(u), O.params(u)
    with impatient() as ctx:
        for _ in range(3):
            o = assert_matches_oracle(ctx.find_groups(pos, ids, p), pos, ids, u)
        assert np.array_equal(cso.cso_fof(ctx.h, pos, ids, o["sigma"], p), o["l0"])
        l1, l2, _ = cso.cso_levels(ctx.h, pos, ids, o["sigma"], o["l0"], p)
    assert np.array_equal(l1, o["l1"]) and np.array_equal(l2, o["l2"])


# 4,096-element list tiles from 2^21 particles on
def test_large_tiles():
    pos, ids, meta = synth.nfw_box(128, 0.4, 20, 20000, seed=92, n_total=2_300_000)
    assert len(pos) > 1 << 21
    p = cso.cso_params_default(meta["u"])
    with cso.Context(0, flags=cso.FLAG_BATCHED) as ctx:
        want = ctx.find_groups(pos, ids, p, on_device=True, radial=True)
    with impatient() as ctx:
        got = ctx.find_groups(pos, ids, p, on_device=True, radial=True)
    for k in want:
        assert np.array_equal(got[k], want[k]), k

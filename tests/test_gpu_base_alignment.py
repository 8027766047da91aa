"""Gradients whose first element lies on a 16- but not on a 32-byte boundary: the same results as from the start of an
allocation, on sizes that are streamed."""
import numpy as np
import pytest
import torch

import ogq_workloads as wl
import paper_2002_11082_b200 as ogq

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_helpers import DeviceBucket

SIZES = [1, 300_007, 16_384, 16_385, 9, 1_000_003, 70_000, 4099]


def bucket(shift):
    """The same bucket with its gradient `shift` elements into an allocation."""
    off = wl.offsets_from_sizes(SIZES)
    v = np.random.Generator(np.random.PCG64(5)).laplace(2e-4, 1e-3, int(off[-1])).astype(np.float32)
    db = DeviceBucket(v, off)
    buf = torch.full((db.N + 16,), float("nan"), device=db.dev)
    buf[shift : shift + db.N] = db.grad
    db.grad = buf[shift : shift + db.N]
    return db


@pytest.mark.parametrize("clip", [False, True])
def test_bingrad_b(clip):
    got = []
    for shift in (0, 4):
        db = bucket(shift)
        if clip:
            tau, st = torch.full((db.T,), 1.5e-3, device=db.dev), torch.zeros(db.T, dtype=torch.int32, device=db.dev)
            lv, th = torch.zeros((db.T, 2), device=db.dev), torch.zeros(db.T, device=db.dev)
            ogq.ogq_levels_bingrad_clipped(db.grad, db.off, db.T, db.N, ogq.OGQ_BINGRAD_B, 1, tau, lv, th, st, db.ws, db.ws_bytes)
            got.append((lv.cpu().numpy(), th.cpu().numpy(), st.cpu().numpy()))
        else:
            got.append(db.levels_bingrad(ogq.OGQ_BINGRAD_B, 1))
    # fp64 sums of the same values in another order: their fp32 roundings are equal or neighbours
    (a_lv, a_th, a_st), (b_lv, b_th, b_st) = got
    assert np.array_equal(a_st, b_st)
    assert np.all(np.abs(a_lv - b_lv) <= 2.0**-22 * np.abs(a_lv)) and np.all(np.abs(a_th - b_th) <= 2.0**-22 * np.abs(a_th))

"""Shares of the streaming CTAs in the exact selection: pieces that end inside a trip, tensors next to the size that is not
streamed, hundreds of those between streamed ones, and more tensors than the shares are worked out for."""
import numpy as np
import pytest
import torch

import oracle
import ogq_workloads as wl
import paper_2002_11082_b200 as ogq

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_helpers import DeviceBucket

BUCKETS = {
    "trips": [8192 * 3, 8192 * 5 + 1, 8192 * 4 - 3, 16385],
    "between": [7, 40_000, 16_384, *[3, 0, 61] * 100, 16_385, *[1] * 70, 130_001, 5, 0],
    "one": [300_007],
    "many": [*[2] * 2500, 20_000, *[3] * 2500, 50_001, 1],  # more than 4096 tensors: equal chunks
}


@pytest.mark.parametrize("bucket", BUCKETS)
def test_levels_of_shares(bucket):
    sizes = BUCKETS[bucket]
    off = wl.offsets_from_sizes(sizes)
    r = np.random.Generator(np.random.PCG64(len(sizes)))
    v = (r.standard_normal(int(off[-1])) * np.exp(r.uniform(-3.0, 3.0, int(off[-1])))).astype(np.float32)
    db = DeviceBucket(v, off)
    got = {"orq": db.levels_orq(9), "pb": db.levels_bingrad(ogq.OGQ_BINGRAD_PB)[::2]}
    want = {"orq": oracle.bucket_levels_orq(v, off, 9), "pb": oracle.bucket_levels_bingrad(v, off, oracle.PB)[::2]}
    for k in got:
        (lv, st), (w_lv, w_st) = got[k], want[k]
        assert np.array_equal(st, w_st)
        if k == "orq":  # order statistics
            assert np.array_equal(lv, w_lv.astype(np.float32))
        assert np.all(np.abs(lv.astype(np.float64) - w_lv) <= 1e-5 * np.max(np.abs(w_lv), axis=1, keepdims=True)), k

"""The exact selection of tensors with more candidates than one CTA's index holds, whose keys are copied in order of
round 1's cells: on both sides of that number, beside tensors that take the other ways, with cells of many equal keys, of few
keys, and of a whole binade."""
import numpy as np
import pytest
import torch

import oracle
import ogq_workloads as wl

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_helpers import DeviceBucket

SIZES = [700_001, 100, 1_400_003, 16_385, 2_800_000, 5_600_001]


def values_of(kind, n, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    v = (r.standard_exponential(n) * np.where(r.random(n) < 0.5, 1.0, -1.0)).astype(np.float32)
    if kind == "ties":  # a few keys to a cell, each many times
        bits = v.view(np.uint32) & np.uint32(0xFFFFE000)
        return bits.view(np.float32)
    if kind == "binades":  # most values far below the fine cells, where a cell is a binade
        v[r.random(n) < 0.9] *= np.float32(1e-9)
        return v
    if kind == "outlier":  # levels in cells that hold a few values of millions
        v[:4] = np.float32([50.0, -70.0, 120.0, -200.0])
        return v
    return v


@pytest.mark.parametrize("kind", ["laplace", "ties", "binades", "outlier"])
def test_levels_from_ordered_cells(kind):
    v = np.concatenate([values_of(kind, n, n) for n in SIZES])
    off = wl.offsets_from_sizes(SIZES)
    db = DeviceBucket(v, off)
    for s in (3, 9, 17):
        lv, st = db.levels_orq(s)
        w_lv, w_st = oracle.bucket_levels_orq(v, off, s)
        assert np.array_equal(st, w_st)
        # levels are values of the data: equal, or the next one where fp64 sums put T on the other side of an integer
        assert np.all(np.abs(lv.astype(np.float64) - w_lv) <= 1e-5 * np.max(np.abs(w_lv), axis=1, keepdims=True)), (kind, s)
        assert np.mean(lv == w_lv) > 0.9, (kind, s)
        again, _ = db.levels_orq(s)
        assert np.array_equal(lv, again)

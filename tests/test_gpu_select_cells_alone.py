"""Tensors whose candidates one CTA selects among cell by cell: on both sides of the fullest cell it takes, alone and beside a
tensor that a cluster works on; cells of one value, of a few, and of values that share their leading bits.  Levels are order
statistics: they are the oracle's bit for bit."""
import numpy as np
import pytest
import torch

import oracle
import ogq_workloads as wl

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_helpers import DeviceBucket


def values_of(kind, n, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    v = (r.standard_exponential(n) * np.where(r.random(n) < 0.5, 1.0, -1.0)).astype(np.float32)
    if kind == "half":  # 8 significant bits: one value to a cell
        return (v.view(np.uint32) & np.uint32(0xFFFF0000)).view(np.float32)
    if kind == "few":  # 3000 values, each hundreds of times
        return np.sort(v)[:: n // 3000][r.integers(0, 3000, n)]
    return v


@pytest.mark.parametrize("kind", ["laplace", "half", "few"])
@pytest.mark.parametrize("sizes", [[1_200_000, 17_000], [4_000_003], [1_500_000, 2_500_001, 9_000_000]])
def test_levels_from_cells_by_one_cta(kind, sizes):
    v = np.concatenate([values_of(kind, n, n) for n in sizes])
    off = wl.offsets_from_sizes(sizes)
    db = DeviceBucket(v, off)
    for s in (3, 9, 17):
        lv, st = db.levels_orq(s)
        w_lv, w_st = oracle.bucket_levels_orq(v, off, s)
        assert np.array_equal(st, w_st)
        assert np.array_equal(lv, w_lv.astype(np.float32)), (kind, s)

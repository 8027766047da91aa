"""The exact selection where its ways part: tensors on both sides of the size that the first solver pass takes alone,
of one chunk and of several, and values that leave few or very many candidate cells."""
import numpy as np
import pytest
import torch

import oracle
import ogq_workloads as wl
import paper_2002_11082_b200 as ogq

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_helpers import DeviceBucket

SIZES = [1023, 8191, 8193, 16383, 16384, 16385, 20001, 65537, 300003]


def values_of(kind, n, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    z = r.standard_normal(n).astype(np.float32)
    if kind == "wide":  # magnitudes over many binades: the level search meets many cells
        return np.sign(z) * np.exp(r.uniform(-60.0, 20.0, n)).astype(np.float32)
    if kind == "peak":  # all values share their leading bits
        return np.float32(1.0) + np.float32(1e-5) * z
    if kind == "flat":  # evenly spread: levels far apart, every candidate cell sparse
        return r.uniform(-1.0, 1.0, n).astype(np.float32)
    v = np.round(z * np.float32(2.0)).astype(np.float32)  # few distinct values, one huge
    v[0] = np.float32(1e6)
    return v


@pytest.mark.parametrize("kind", ["wide", "peak", "flat", "few"])
def test_levels_at_the_edges(kind):
    v = np.concatenate([values_of(kind, n, n) for n in SIZES])
    off = wl.offsets_from_sizes(SIZES)
    db = DeviceBucket(v, off)
    for s in (3, 17):
        lv, st = db.levels_orq(s)
        w_lv, w_st = oracle.bucket_levels_orq(v, off, s)
        assert np.array_equal(st, w_st)
        assert np.all(np.abs(lv.astype(np.float64) - w_lv) <= 1e-5 * np.max(np.abs(w_lv), axis=1, keepdims=True)), (kind, s)
    lv, _, st = db.levels_bingrad(ogq.OGQ_BINGRAD_PB)
    w_lv, _, w_st = oracle.bucket_levels_bingrad(v, off, oracle.PB)
    assert np.array_equal(st, w_st)
    assert np.all(np.abs(lv.astype(np.float64) - w_lv) <= 1e-5 * np.max(np.abs(w_lv), axis=1, keepdims=True)), kind

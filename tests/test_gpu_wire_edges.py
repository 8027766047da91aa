"""Quantizer and server step where their loops part: tensors of less and more than the groups of one trip, tensors that
do not start on a 16-byte boundary, partial groups, levels outside the range of the scaled rounding decision, and
worker counts around those that a table of sums takes in."""
import numpy as np
import pytest
import torch

import oracle
import ogq_workloads as wl
import paper_2002_11082_b200 as ogq

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_helpers import DeviceBucket

SIZES = [1, 255, 257, 1024, 1281, 4097, 8195, 3, 12801, 40962, 70000]  # starts at every offset from a 16-byte boundary


def levels_of(s, scale):
    lv = np.stack([np.linspace(-2.0, 2.0, s) * (1 + t % 3) for t in range(len(SIZES))])
    return (lv * scale).astype(np.float32)


def values(seed, scale):
    r = np.random.Generator(np.random.PCG64(seed))
    return (r.standard_normal(sum(SIZES)) * scale).astype(np.float32)


@pytest.mark.parametrize("scale", [1e-3, 2.0**110, 2.0**-110])
@pytest.mark.parametrize("s", [2, 3, 5, 9, 17])
def test_quantize_edges(s, scale):
    v, off = values(s, scale), wl.offsets_from_sizes(SIZES)
    db = DeviceBucket(v, off)
    lv = levels_of(s, scale)
    want, _ = oracle.bucket_quantize_pack(v, off, oracle.ORQ if s > 2 else oracle.PB, s, lv, None, 11, 4)
    got, _ = db.quantize_pack(ogq.OGQ_ORQ if s > 2 else ogq.OGQ_BINGRAD_PB, s, lv, None, 11, 4)
    assert np.array_equal(got, want)


@pytest.mark.parametrize("K", [1, 4, 7, 8, 9, 16])
@pytest.mark.parametrize("s", [2, 3, 5, 9, 17])
def test_unpack_sum_edges(s, K):
    off = wl.offsets_from_sizes(SIZES)
    db = DeviceBucket(values(1, 1.0), off)
    packed, levels = [], []
    for k in range(K):
        lv = levels_of(s, 1.0 + 0.37 * k)
        pk, _ = oracle.bucket_quantize_pack(values(k, 1.0), off, oracle.ORQ if s > 2 else oracle.PB, s, lv, None, 1, k)
        packed.append(pk)
        levels.append(lv)
    want = oracle.bucket_unpack_sum(packed, levels, off, s, 1.0 / K)
    got = db.unpack_sum(packed, levels, s, 1.0 / K)
    for a, e in zip(off[:-1], off[1:]):
        assert np.all(np.abs(got[a:e].astype(np.float64) - want[a:e]) <= 1e-5 * np.max(np.abs(want[a:e])))

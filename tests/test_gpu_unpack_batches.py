"""Server step with more tensors in a CTA's chunk than it keeps level rows for at a time: tensors of a few elements
to a few groups, empty ones among them, for worker counts that change how many rows fit."""
import numpy as np
import pytest
import torch

import oracle
import ogq_workloads as wl

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_helpers import DeviceBucket


@pytest.mark.parametrize("K", [1, 3, 8, 33, 64])
@pytest.mark.parametrize("s", [2, 3, 5, 9, 17])
def test_unpack_sum_many_small_tensors(s, K):
    r = np.random.Generator(np.random.PCG64(s * 100 + K))
    sizes = np.concatenate([r.integers(0, 40, 70), r.integers(200, 900, 30), [5000], r.integers(1, 9, 40)]).astype(np.int64)
    off, T = wl.offsets_from_sizes(sizes), sizes.size
    n = int(off[-1])
    packed, levels = [], []
    for k in range(K):
        lv = np.sort(r.standard_normal((T, s)).astype(np.float32), axis=1)
        v = r.standard_normal(n).astype(np.float32)
        pk, _ = oracle.bucket_quantize_pack(v, off, oracle.ORQ if s > 2 else oracle.PB, s, lv, None, 1, k)
        packed.append(pk)
        levels.append(lv)
    db = DeviceBucket(np.zeros(n, np.float32), off)
    got = db.unpack_sum(packed, levels, s, 1.0 / K)
    want = np.asarray(oracle.bucket_unpack_sum(packed, levels, off, s, 1.0 / K))
    # fp32 sums of K terms in one order: at most K roundings of 2^-24 of the largest partial sum
    bound = K * 2.0**-24 * np.max([np.max(np.abs(l)) for l in levels])
    assert np.all(np.abs(got.astype(np.float64) - want) <= bound)

"""Segments with nothing, or with equal values, between their two levels, where T of the discrete condition is an integer: the
level is the lower end whatever the order in which values reach their cells."""
import numpy as np
import pytest
import torch

import oracle
import ogq_workloads as wl

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_helpers import DeviceBucket


@pytest.mark.parametrize("seed", range(3))
def test_few_values_per_segment(seed):
    r = np.random.Generator(np.random.PCG64(seed))
    sizes = [int(n) for n in r.integers(3, 130, 150)] + [17_000, 20_000]
    v = (r.standard_exponential(sum(sizes)) * np.where(r.random(sum(sizes)) < 0.5, 1.0, -1.0)).astype(np.float32)
    v[r.random(v.size) < 0.8] *= np.float32(1e-9)
    off = wl.offsets_from_sizes(sizes)
    db = DeviceBucket(v, off)
    for s in (9, 17):
        want, _ = oracle.bucket_levels_orq(v, off, s)
        for _ in range(12):
            lv, _ = db.levels_orq(s)
            assert np.array_equal(lv, want), np.argwhere(lv != want)[:4]

"""The sort of the fixed-length buckets where it can go wrong: the shortest and longest buckets of every
team size, lengths that do not fill the team, a ragged last bucket, and values the cells do not separate
(a narrow peak far from zero, a few distinct values, mostly zeros, one huge outlier)."""
import numpy as np
import pytest
import torch

from test_gpu_buckets import check_against_oracle

pytestmark = pytest.mark.gpu


def values_of(kind, n, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    z = rng.standard_normal(n, dtype=np.float32)
    if kind == "peak":  # distinct values that share their leading bits: the network of last resort
        return np.float32(1.0) + np.float32(1e-4) * z
    if kind == "few":
        return np.round(z * np.float32(1.5)).astype(np.float32)
    if kind == "zeros":
        return np.where(rng.random(n) < 0.8, np.float32(-0.0), z).astype(np.float32)
    v = z * np.float32(1e-3)  # outlier
    v[:: max(1, n // 5)] = np.float32(50.0)
    return v


@pytest.mark.parametrize("kind", ["peak", "few", "zeros", "outlier"])
@pytest.mark.parametrize("d", [128, 256, 384, 512, 640, 4096, 4224, 8192, 16384, 32768])
def test_sort_edges(d, kind):
    v = values_of(kind, 3 * d + 77, d)
    check_against_oracle(v, d, "orq", 9)
    check_against_oracle(v, d, "pb", 2)

"""Server step of one worker against the general one: with a second worker whose levels are all zero the sums are the
same values, bit for bit.  Codes are random words, so those that no quantizer writes (s and above) are among them."""
import numpy as np
import pytest
import torch

import ogq_workloads as wl
import paper_2002_11082_b200 as ogq

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_helpers import DeviceBucket

# a group, a warp's trip of two and four groups, a CTA's trips, one element less or more; starts off a 16-byte boundary
EDGES = [1, 255, 256, 257, 0, 2047, 2049, 4096, 4095, 8193, 3, 16385, 32767, 70001]


@pytest.mark.parametrize("sizes", [[1], EDGES, [9_000_001] + EDGES], ids=["one", "edges", "long"])
@pytest.mark.parametrize("s", [2, 3, 5, 9, 17])
def test_one_worker_is_the_general_sum(s, sizes):
    r = np.random.Generator(np.random.PCG64(s))
    off = wl.offsets_from_sizes(sizes)
    T = len(sizes)
    words = int(ogq.ogq_packed_layout(off, ogq.ogq_bits_for_levels(s))[-1])
    codes = r.integers(0, 2**32, words, dtype=np.uint32)
    lv = np.sort(r.standard_normal((T, s)).astype(np.float32), axis=1)
    lv[0, 0], lv[-1, 0], lv[T // 2, -1] = -0.0, -np.inf, np.inf
    db = DeviceBucket(np.zeros(int(off[-1]), np.float32), off)
    one = db.unpack_sum([codes], [lv], s, 0.37)
    two = db.unpack_sum([codes, codes], [lv, np.zeros_like(lv)], s, 0.37)
    assert np.array_equal(one.view(np.uint32), two.view(np.uint32))

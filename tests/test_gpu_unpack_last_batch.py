"""Server steps whose last batch of workers is a full one, alone and behind others: the sums of the server step, of the one for
fixed-length buckets (at an odd total) and of one-bit codes up to twice the table's workers, as fp32 additions in worker order."""
import numpy as np
import pytest
import torch

import ogq_workloads as wl
import paper_2002_11082_b200 as ogq

pytestmark = pytest.mark.gpu

SIZES = [2052, 4096, 20, 776, 3, 1033, 12_300, 70_001]


@pytest.mark.parametrize("K", [4, 8, 13, 16, 17, 20, 24, 33])
@pytest.mark.parametrize("s", [2, 3, 5, 9, 17])
def test_sums_in_worker_order(s, K):
    dev, bits, total, d = torch.device("cuda:0"), ogq.ogq_bits_for_levels(s), sum(SIZES), 512
    g = torch.Generator(device=dev)
    g.manual_seed(100 * s + K)
    scale = 0.5
    for h_off in (wl.offsets_from_sizes(SIZES), np.minimum(np.arange(-(-total // d) + 1, dtype=np.int64) * d, total)):
        T = h_off.size - 1
        h_po = ogq.ogq_packed_layout(h_off, bits)
        pk = [torch.randint(-(2**31), 2**31 - 1, (int(h_po[-1]),), dtype=torch.int32, device=dev, generator=g) for _ in range(K)]
        lv = [torch.randn((T, s), device=dev, generator=g) for _ in range(K)]
        pk_p, lv_p = ogq.device_pointer_array(pk), ogq.device_pointer_array(lv)
        want = torch.zeros(total, device=dev)
        for t in range(T):
            a, e = int(h_off[t]), int(h_off[t + 1])
            i = torch.arange(e - a, device=dev) * bits
            w, sh, last = int(h_po[t]) + i // 32, i % 32, int(h_po[-1]) - 1
            for k in range(K):  # codes above s - 1 stand for the top level
                words = (pk[k][w].long() & 0xFFFFFFFF) | (pk[k][(w + 1).clamp(max=last)].long() & 0xFFFFFFFF) << 32
                want[a:e] += lv[k][t][((words >> sh) & ((1 << bits) - 1)).clamp(max=s - 1)]
        want *= scale
        got = torch.full((total,), 5.0, device=dev)
        ogq.ogq_unpack_sum(pk_p, lv_p, K, torch.from_numpy(h_off).to(dev), torch.from_numpy(h_po).to(dev), T, total, s, scale, got)
        assert torch.equal(got, want)
        if T != len(SIZES):
            got.fill_(6.0)
            ogq.ogq_bucket_decode_sum(pk_p, lv_p, K, total, d, s, scale, got)
            assert torch.equal(got, want)

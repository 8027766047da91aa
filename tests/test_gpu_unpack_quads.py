"""Server step for 1-bit codes with four groups of a tensor at a time: every remainder of groups and elements, outputs on and off
16-byte boundaries, worker counts on both sides of four and eight; against the sums in worker order that torch makes."""
import numpy as np
import pytest
import torch

import paper_2002_11082_b200 as ogq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [2, 4, 5, 8, 9])
@pytest.mark.parametrize("sizes", [[5_000_003], [2_600_000, 1_300_021, 999, 2_200_512], [6_000_128, 256 * 9000]])
def test_unpack_sum_of_one_bit_codes(K, sizes):
    dev, T, total = torch.device("cuda:0"), len(sizes), sum(sizes)
    h_off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    h_po = ogq.ogq_packed_layout(h_off, 1)
    g = torch.Generator(device=dev)
    g.manual_seed(K)
    pk = [torch.randint(-(2**31), 2**31 - 1, (int(h_po[-1]),), dtype=torch.int32, device=dev, generator=g) for _ in range(K)]
    lv = [torch.randn((T, 2), device=dev, generator=g) for _ in range(K)]
    out = torch.full((total,), 5.0, device=dev)
    ogq.ogq_unpack_sum(ogq.device_pointer_array(pk), ogq.device_pointer_array(lv), K, torch.from_numpy(h_off).to(dev),
                       torch.from_numpy(h_po).to(dev), T, total, 2, 0.25, out)
    for t, n in enumerate(sizes):
        i = torch.arange(n, device=dev)
        want = torch.zeros(n, device=dev)
        for k in range(K):
            codes = (pk[k][int(h_po[t]) + i // 32] >> (i % 32)) & 1
            want = want + lv[k][t][codes.long()]  # fp32, in worker order
        assert torch.equal(out[int(h_off[t]) : int(h_off[t + 1])], want * 0.25)

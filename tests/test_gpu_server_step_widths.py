"""Server steps at every number of workers of their last, partial batch, with outputs on 16- but not on 32-byte boundaries; the
bucket kernel with one and with two groups at a time; the dense kernel on both sides of the worker counts whose tables of one,
two and three digits fit."""
import numpy as np
import pytest
import torch

import oracle
import ogq_workloads as wl
import paper_2002_11082_b200 as ogq

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_helpers import DeviceBucket

SIZES = [2052, 4096, 20, 776, 3, 1033, 12_300, 8]  # the first tensors begin at offsets of 4, not of 8 elements


def workers(s, K, dense=False):
    off = wl.offsets_from_sizes(SIZES)
    r = np.random.Generator(np.random.PCG64(100 * s + K))
    packed, levels, po = [], [], None
    for k in range(K):
        lv = np.sort(r.standard_normal((len(SIZES), s)).astype(np.float32), axis=1)
        v = r.standard_normal(int(off[-1])).astype(np.float32)
        pk, po, codes = oracle.bucket_quantize_pack(v, off, oracle.ORQ if s > 2 else oracle.PB, s, lv, None, 1, k, return_codes=True)
        if dense:
            pk, po = oracle.bucket_pack_dense(codes, off, s)
        packed.append(pk)
        levels.append(lv)
    # fp32 sums of K terms: at most K roundings of 2^-24 of the largest partial sum, and one of the product
    bound = (K + 1) * 2.0**-24 * np.max([np.max(np.abs(l)) for l in levels])
    return off, packed, levels, po, bound


@pytest.mark.parametrize("K", [2, 3, 5, 6, 7, 10, 12, 15])
@pytest.mark.parametrize("s", [2, 3, 5, 9, 17])
def test_unpack_sum_partial_batches(s, K):
    off, packed, levels, _, bound = workers(s, K)
    got = DeviceBucket(np.zeros(int(off[-1]), np.float32), off).unpack_sum(packed, levels, s, 1.0 / K)
    want = np.asarray(oracle.bucket_unpack_sum(packed, levels, off, s, 1.0 / K))
    assert np.all(np.abs(got.astype(np.float64) - want) <= bound)


@pytest.mark.parametrize("s,K", [(3, 10), (3, 11), (3, 48), (3, 49), (5, 1), (5, 20), (5, 21), (9, 6), (17, 7)]
                         + [(s, K) for s in (3, 5, 9, 17) for K in (2, 3, 4, 5, 8)])
def test_unpack_sum_dense_tables(s, K):
    off, packed, levels, h_po, bound = workers(s, K, dense=True)
    dev = torch.device("cuda:0")
    d_pk = [torch.from_numpy(p.view(np.int32)).to(dev) for p in packed]
    d_lv = [torch.from_numpy(l).to(dev) for l in levels]
    out = torch.full((int(off[-1]),), 12345.0, device=dev)
    ogq.ogq_unpack_sum_dense(ogq.device_pointer_array(d_pk), ogq.device_pointer_array(d_lv), K, torch.from_numpy(off).to(dev),
                             torch.from_numpy(h_po).to(dev), len(SIZES), int(off[-1]), s, 1.0 / K, out)
    want = oracle.bucket_unpack_sum_dense(packed, levels, off, s, 1.0 / K)
    assert np.all(np.abs(out.cpu().numpy().astype(np.float64) - want) <= bound)


@pytest.mark.parametrize("s,d,K,total", [(9, 512, 3, 11_000_077), (3, 640, 2, 10_500_001), (5, 4096, 6, 9_800_000), (2, 1024, 9, 12_345_679),
                                         (17, 256, 5, 10_000_001), (9, 512, 7, 900_013), (2, 2048, 1, 11_000_077)])
def test_bucket_decode_sum_runs(s, d, K, total):
    """Equal to ogq_unpack_sum called with offsets j * d, bit for bit: the same additions (any words are codes)."""
    dev, bits = torch.device("cuda:0"), ogq.ogq_bits_for_levels(s)
    T = -(-total // d)
    g = torch.Generator(device=dev)
    g.manual_seed(total)
    words = ogq.ogq_bucket_packed_words(total, d, bits)
    d_pk = [torch.randint(-(2**31), 2**31 - 1, (words,), dtype=torch.int32, device=dev, generator=g) for _ in range(K)]
    d_lv = [torch.randn((T, s), device=dev, generator=g).sort(dim=1)[0].contiguous() for _ in range(K)]
    h_off = np.minimum(np.arange(T + 1, dtype=np.int64) * d, total)
    off, po = torch.from_numpy(h_off).to(dev), torch.from_numpy(ogq.ogq_packed_layout(h_off, bits)).to(dev)
    a, b = torch.full((total,), 1.0, device=dev), torch.full((total,), 2.0, device=dev)
    pk, lv = ogq.device_pointer_array(d_pk), ogq.device_pointer_array(d_lv)
    ogq.ogq_bucket_decode_sum(pk, lv, K, total, d, s, 1.0 / K, a)
    ogq.ogq_unpack_sum(pk, lv, K, off, po, T, total, s, 1.0 / K, b)
    assert torch.equal(a, b)

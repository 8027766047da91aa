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


@pytest.mark.parametrize("K", [1, 4, 5, 11])
@pytest.mark.parametrize("s", [3, 5, 9, 17])
def test_dense_wire_edges(s, K):
    off = wl.offsets_from_sizes(SIZES)
    packed, levels = [], []
    for k in range(K):
        v, lv = values(k, 1.0), levels_of(s, 1.0 + 0.37 * k)
        _, _, codes = oracle.bucket_quantize_pack(v, off, oracle.ORQ, s, lv, None, 11, k, return_codes=True)
        pk, h_po = oracle.bucket_pack_dense(codes, off, s)
        packed.append(pk)
        levels.append(lv)
    db = DeviceBucket(values(0, 1.0), off)
    po = torch.from_numpy(h_po).to(db.dev)
    got = torch.zeros(int(h_po[-1]), dtype=torch.int32, device=db.dev)
    d_lv = [torch.from_numpy(lv).to(db.dev) for lv in levels]
    ogq.ogq_quantize_pack_dense(db.grad, db.off, db.T, db.N, s, d_lv[0], 11, 0, po, got)
    assert np.array_equal(got.cpu().numpy().view(np.uint32), packed[0])
    d_pk = [torch.from_numpy(p.view(np.int32)).to(db.dev) for p in packed]
    out = torch.empty(db.N, device=db.dev)
    ogq.ogq_unpack_sum_dense(ogq.device_pointer_array(d_pk), ogq.device_pointer_array(d_lv), K, db.off, po, db.T, db.N, s,
                             1.0 / K, out)
    h, want = out.cpu().numpy().astype(np.float64), oracle.bucket_unpack_sum_dense(packed, levels, off, s, 1.0 / K)
    for a, e in zip(off[:-1], off[1:]):
        assert np.all(np.abs(h[a:e] - want[a:e]) <= 1e-5 * np.max(np.abs(want[a:e])))


@pytest.mark.parametrize("c", [0.0, 1.7])
@pytest.mark.parametrize("sizes", [[65537, 65535], [131073], [16383, 0, 16384, 16385, 1, 100003]])
def test_bingrad_b_edges(sizes, c):
    """One cluster launch up to 131072 elements, CTAs of their own for tensors of up to 16384, the flat passes."""
    r = np.random.Generator(np.random.PCG64(len(sizes)))
    v, off = (r.laplace(size=sum(sizes)) * 1e-3 + 2e-4).astype(np.float32), wl.offsets_from_sizes(sizes)
    db = DeviceBucket(v, off)
    lv, th = torch.zeros((db.T, 2), device=db.dev), torch.zeros(db.T, device=db.dev)
    st, tau = torch.zeros(db.T, dtype=torch.int32, device=db.dev), torch.zeros(db.T, device=db.dev)
    for lloyd in (0, 2):
        if c:
            ogq.ogq_clip_threshold(db.grad, db.off, db.T, db.N, c, tau, st, db.ws, db.ws_bytes)
            w_tau, _ = oracle.bucket_clip_thresholds(v, off, c)
            assert np.allclose(tau.cpu().numpy(), w_tau, rtol=1e-6, atol=0.0)
            ogq.ogq_levels_bingrad_clipped(db.grad, db.off, db.T, db.N, ogq.OGQ_BINGRAD_B, lloyd, tau, lv, th, st, db.ws, db.ws_bytes)
            x = oracle.bucket_clip(v, off, tau.cpu().numpy())
        else:
            ogq.ogq_levels_bingrad(db.grad, db.off, db.T, db.N, ogq.OGQ_BINGRAD_B, lloyd, lv, th, st, db.ws, db.ws_bytes)
            x = v
        w_lv, w_th, w_st = oracle.bucket_levels_bingrad(x, off, oracle.B, lloyd)
        assert np.array_equal(st.cpu().numpy(), w_st)
        tol = 1e-5 * np.max(np.abs(w_lv), axis=1, keepdims=True)
        assert np.all(np.abs(lv.cpu().numpy().astype(np.float64) - w_lv) <= tol)
        assert np.all(np.abs(th.cpu().numpy().astype(np.float64) - w_th) <= tol[:, 0])

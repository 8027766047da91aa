"""Clipped selection with any share of the values at the threshold: none, a few, most, all of them, and thresholds outside round
1's fine cells; heavy magnitudes in one cell without clipping."""
import numpy as np
import pytest
import torch

import oracle
import ogq_workloads as wl
import paper_2002_11082_b200 as ogq

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_helpers import DeviceBucket

SIZES = [200_003, 70_000, 300_001, 16_385, 100_000, 5000, 150_000]
TAU = [0.7, 1e9, 1e-3, 0.0, 1e-12, 0.5, 2.2]


@pytest.mark.parametrize("shape", ["normal", "uniform"])
def test_clipped_levels_with_any_threshold(shape):
    r = np.random.Generator(np.random.PCG64(len(shape)))
    n = sum(SIZES)
    v = (r.standard_normal(n) if shape == "normal" else r.uniform(-1.0, 1.0, n)).astype(np.float32)
    off, tau = wl.offsets_from_sizes(SIZES), np.array(TAU, np.float32)
    x = oracle.bucket_clip(v, off, tau)
    db = DeviceBucket(v, off)
    d_tau, st = torch.from_numpy(tau).to(db.dev), torch.zeros(db.T, dtype=torch.int32, device=db.dev)
    for s in (3, 9):
        lv = torch.zeros((db.T, s), device=db.dev)
        ogq.ogq_levels_orq_clipped(db.grad, db.off, db.T, db.N, s, d_tau, lv, st, db.ws, db.ws_bytes)
        w_lv, w_st = oracle.bucket_levels_orq(x, off, s)
        assert np.array_equal(st.cpu().numpy(), w_st)
        assert np.array_equal(lv.cpu().numpy(), w_lv.astype(np.float32)), s  # order statistics
    lv, th = torch.zeros((db.T, 2), device=db.dev), torch.zeros(db.T, device=db.dev)
    ogq.ogq_levels_bingrad_clipped(db.grad, db.off, db.T, db.N, ogq.OGQ_BINGRAD_PB, 0, d_tau, lv, th, st, db.ws, db.ws_bytes)
    w_lv, _, w_st = oracle.bucket_levels_bingrad(x, off, oracle.PB)
    assert np.array_equal(st.cpu().numpy(), w_st)
    assert np.all(np.abs(lv.cpu().numpy().astype(np.float64) - w_lv) <= 1e-5 * np.max(np.abs(w_lv), axis=1, keepdims=True))
    lv, _, st = db.levels_bingrad(ogq.OGQ_BINGRAD_PB)
    w_lv, _, w_st = oracle.bucket_levels_bingrad(v, off, oracle.PB)
    assert np.array_equal(st, w_st) and np.all(np.abs(lv.astype(np.float64) - w_lv) <= 1e-5 * np.max(np.abs(w_lv), axis=1, keepdims=True))


def test_thresholds_that_the_library_does_not_make():
    """A caller's threshold that is not a number, infinite or negative: copysign(min(|v|, tau), v) with the minimum of IEEE 754,
    which passes a NaN over."""
    tau = np.array([np.nan, np.inf, -0.5, np.nan, -1e-3, np.nan, np.inf], np.float32)
    r = np.random.Generator(np.random.PCG64(9))
    v, off = r.standard_normal(sum(SIZES)).astype(np.float32), wl.offsets_from_sizes(SIZES)
    x = np.concatenate([np.copysign(np.fmin(np.abs(v[a:e]), t), v[a:e]) for a, e, t in zip(off[:-1], off[1:], tau)]).astype(np.float32)
    db = DeviceBucket(v, off)
    d_tau, st = torch.from_numpy(tau).to(db.dev), torch.zeros(db.T, dtype=torch.int32, device=db.dev)
    for s in (3, 9):
        lv = torch.zeros((db.T, s), device=db.dev)
        ogq.ogq_levels_orq_clipped(db.grad, db.off, db.T, db.N, s, d_tau, lv, st, db.ws, db.ws_bytes)
        w_lv, w_st = oracle.bucket_levels_orq(x, off, s)
        assert np.array_equal(st.cpu().numpy(), w_st)
        assert np.array_equal(lv.cpu().numpy(), w_lv.astype(np.float32)), s
    d_tau = d_tau.abs()  # (magnitudes are not negative)
    x = np.concatenate([np.copysign(np.fmin(np.abs(v[a:e]), np.abs(t)), v[a:e]) for a, e, t in zip(off[:-1], off[1:], tau)]).astype(np.float32)
    lv, th = torch.zeros((db.T, 2), device=db.dev), torch.zeros(db.T, device=db.dev)
    ogq.ogq_levels_bingrad_clipped(db.grad, db.off, db.T, db.N, ogq.OGQ_BINGRAD_PB, 0, d_tau, lv, th, st, db.ws, db.ws_bytes)
    w_lv, _, w_st = oracle.bucket_levels_bingrad(x, off, oracle.PB)
    assert np.array_equal(st.cpu().numpy(), w_st)
    assert np.all(np.abs(lv.cpu().numpy().astype(np.float64) - w_lv) <= 1e-5 * np.max(np.abs(w_lv), axis=1, keepdims=True))

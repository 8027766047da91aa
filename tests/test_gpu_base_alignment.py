"""Gradients and outputs whose first element lies on a 16- but not on a 32-byte boundary: the same results as from the start of
an allocation, on sizes that are streamed."""
import numpy as np
import pytest
import torch

import ogq_workloads as wl
import paper_2002_11082_b200 as ogq

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_helpers import DeviceBucket

SIZES = [1, 300_007, 16_384, 16_385, 9, 1_000_003, 70_000, 4099]


def bucket(shift):
    """The same bucket with its gradient `shift` elements into an allocation."""
    off = wl.offsets_from_sizes(SIZES)
    v = np.random.Generator(np.random.PCG64(5)).laplace(2e-4, 1e-3, int(off[-1])).astype(np.float32)
    db = DeviceBucket(v, off)
    buf = torch.full((db.N + 16,), float("nan"), device=db.dev)
    buf[shift : shift + db.N] = db.grad
    db.grad = buf[shift : shift + db.N]
    return db


@pytest.mark.parametrize("clip", [False, True])
def test_bingrad_b(clip):
    got = []
    for shift in (0, 4):
        db = bucket(shift)
        if clip:
            tau, st = torch.full((db.T,), 1.5e-3, device=db.dev), torch.zeros(db.T, dtype=torch.int32, device=db.dev)
            lv, th = torch.zeros((db.T, 2), device=db.dev), torch.zeros(db.T, device=db.dev)
            ogq.ogq_levels_bingrad_clipped(db.grad, db.off, db.T, db.N, ogq.OGQ_BINGRAD_B, 1, tau, lv, th, st, db.ws, db.ws_bytes)
            got.append((lv.cpu().numpy(), th.cpu().numpy(), st.cpu().numpy()))
        else:
            got.append(db.levels_bingrad(ogq.OGQ_BINGRAD_B, 1))
    # fp64 sums of the same values in another order: their fp32 roundings are equal or neighbours
    (a_lv, a_th, a_st), (b_lv, b_th, b_st) = got
    assert np.array_equal(a_st, b_st)
    assert np.all(np.abs(a_lv - b_lv) <= 2.0**-22 * np.abs(a_lv)) and np.all(np.abs(a_th - b_th) <= 2.0**-22 * np.abs(a_th))


@pytest.mark.parametrize("clip", [False, True])
def test_selection_and_codes(clip):
    """Levels of ORQ and the codes are the same bit for bit; BinGrad-pb's level comes from fp64 sums in another order."""
    a, b = bucket(0), bucket(4)
    tau = torch.full((a.T,), 1.5e-3, device=a.dev)
    for s in (3, 9, 17):
        got = []
        for db in (a, b):
            lv, st = torch.zeros((db.T, s), device=db.dev), torch.zeros(db.T, dtype=torch.int32, device=db.dev)
            if clip:
                ogq.ogq_levels_orq_clipped(db.grad, db.off, db.T, db.N, s, tau, lv, st, db.ws, db.ws_bytes)
            else:
                ogq.ogq_levels_orq(db.grad, db.off, db.T, db.N, s, lv, st, db.ws, db.ws_bytes)
            h = lv.cpu().numpy()
            got.append((h, st.cpu().numpy(), db.quantize_pack(ogq.OGQ_ORQ, s, h, None, 3, 1, tau=tau if clip else None)[0]))
        assert all(np.array_equal(x, y) for x, y in zip(*got)), s
    if not clip:
        (a_lv, _, a_st), (b_lv, _, b_st) = (db.levels_bingrad(ogq.OGQ_BINGRAD_PB) for db in (a, b))
        assert np.array_equal(a_st, b_st) and np.all(np.abs(a_lv - b_lv) <= 2.0**-22 * np.abs(a_lv))


@pytest.mark.parametrize("s", [2, 3, 5, 9, 17])
def test_server_steps(s):
    """The sums are fp32 additions in worker order: bit for bit the same wherever the output begins."""
    db, K, d, bits = bucket(0), 5, 512, ogq.ogq_bits_for_levels(s)
    g = torch.Generator(device=db.dev)
    g.manual_seed(s)
    h_off = np.minimum(np.arange(-(-db.N // d) + 1, dtype=np.int64) * d, db.N)
    wire = {"bits": ogq.ogq_packed_layout(db.h_off, bits), "buckets": ogq.ogq_packed_layout(h_off, bits)}
    if s > 2:
        wire["dense"] = ogq.ogq_dense_layout(db.h_off, s)
    for kind, h_po in wire.items():
        T = h_po.size - 1
        pk = [torch.randint(0, s**ogq.ogq_dense_digits(s) if kind == "dense" else 2**31 - 1, (int(h_po[-1]),), device=db.dev,
                            generator=g).to(torch.int32) for _ in range(K)]
        lv = [torch.randn((T, s), device=db.dev, generator=g) for _ in range(K)]
        pk_p, lv_p, po = ogq.device_pointer_array(pk), ogq.device_pointer_array(lv), torch.from_numpy(h_po).to(db.dev)
        got = []
        for shift in (0, 4):
            buf = torch.full((db.N + 16,), 7.0, device=db.dev)
            out = buf[shift : shift + db.N]
            if kind == "bits":
                ogq.ogq_unpack_sum(pk_p, lv_p, K, db.off, po, T, db.N, s, 0.25, out)
            elif kind == "dense":
                ogq.ogq_unpack_sum_dense(pk_p, lv_p, K, db.off, po, T, db.N, s, 0.25, out)
            else:
                ogq.ogq_bucket_decode_sum(pk_p, lv_p, K, db.N, d, s, 0.25, out)
            assert torch.all(buf[:shift] == 7.0) and torch.all(buf[shift + db.N :] == 7.0)
            got.append(out.clone())
        assert torch.equal(*got), kind

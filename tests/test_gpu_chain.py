"""Launches that begin before the one before them has ended: an average that the server step has just written is encoded again, in
place, again and again on one stream.  Equal bit for bit to the same with a synchronisation after every call."""
import numpy as np
import pytest
import torch

import ogq_workloads as wl
import paper_2002_11082_b200 as ogq

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_helpers import DeviceBucket

BUCKETS = {
    "mixed": [*[3000, 64, 16_000] * 20, 400_003, 50_000, 17, 1_300_001],
    "streamed": [2_000_000, 300_001],
    "small": [4000, 12_000],
    "tiny beside one": [*[64] * 200, 200_000],
}


@pytest.mark.parametrize("clip", [0.0, 2.5])
@pytest.mark.parametrize("scheme,s", [("orq", 3), ("orq", 9), ("pb", 2), ("b", 2)])
@pytest.mark.parametrize("sizes", BUCKETS)
def test_encode_of_an_average_just_written(sizes, scheme, s, clip):
    off = wl.offsets_from_sizes(BUCKETS[sizes])
    v = np.random.Generator(np.random.PCG64(len(sizes))).laplace(0.0, 1e-3, int(off[-1])).astype(np.float32)
    kind = {"orq": ogq.OGQ_ORQ, "pb": ogq.OGQ_BINGRAD_PB, "b": ogq.OGQ_BINGRAD_B}[scheme]
    h_po = ogq.ogq_packed_layout(off, ogq.ogq_bits_for_levels(s))

    def run(wait):
        db = DeviceBucket(v, off)
        po = torch.from_numpy(h_po).to(db.dev)
        lv, th = torch.zeros((db.T, s), device=db.dev), torch.zeros(db.T, device=db.dev)
        tau, st = torch.zeros(db.T, device=db.dev), torch.zeros(db.T, dtype=torch.int32, device=db.dev)
        pk, own = torch.zeros(int(h_po[-1]), dtype=torch.int32, device=db.dev), torch.zeros(int(h_po[-1]), dtype=torch.int32, device=db.dev)
        first = torch.zeros((db.T, s), device=db.dev)
        both, both_lv = ogq.device_pointer_array([pk, own]), ogq.device_pointer_array([lv, first])
        seen = []
        pause = torch.cuda.synchronize if wait else (lambda: None)
        for i in range(8):
            if clip:
                ogq.ogq_clip_threshold(db.grad, db.off, db.T, db.N, clip, tau, st, db.ws, db.ws_bytes)
                pause()
            if scheme == "orq":
                args = (db.grad, db.off, db.T, db.N, s) + ((tau,) if clip else ())
                (ogq.ogq_levels_orq_clipped if clip else ogq.ogq_levels_orq)(*args, lv, st, db.ws, db.ws_bytes)
            else:
                args = (db.grad, db.off, db.T, db.N, kind, 0) + ((tau,) if clip else ())
                (ogq.ogq_levels_bingrad_clipped if clip else ogq.ogq_levels_bingrad)(*args, lv, th, st, db.ws, db.ws_bytes)
            pause()
            if clip:
                ogq.ogq_quantize_pack_clipped(db.grad, db.off, db.T, db.N, kind, s, lv, th, tau, 7 + i, 0, po, pk)
            else:
                ogq.ogq_quantize_pack(db.grad, db.off, db.T, db.N, kind, s, lv, th, 7 + i, 0, po, pk)
            pause()
            if i == 0:  # a second worker, with the codes of the first step
                own.copy_(pk)
                first.copy_(lv)
            seen.append((lv.clone(), st.clone(), pk.clone()))
            pause()
            # the gradient becomes a weighted sum of the two workers' values: other values at every step
            ogq.ogq_unpack_sum(both, both_lv, 2, db.off, po, db.T, db.N, s, 0.5 + 0.25 * (i % 3), db.grad)
            pause()
        torch.cuda.synchronize()
        return seen, db.grad.clone()

    (a, a_grad), (b, b_grad) = run(False), run(True)
    for x, y in zip(a, b):
        assert all(torch.equal(p, q) for p, q in zip(x, y))
    assert torch.equal(a_grad, b_grad)

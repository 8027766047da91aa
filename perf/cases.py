"""The calls whose speed matters to a user of this library, as cases that can be timed.

A case is one worker's or server's share of a data-parallel step on one GPU:

  op "encode"  levels, then quantize + pack, of the worker's own gradient;
  op "decode"  unpack + dequantize + sum of the packed codes of K workers (the broadcast average);
  op "step"    encode of the own gradient, then decode of the K workers' codes, the own ones among them.

Keys of a case:

  layout   "resnet50" / "vgg19": the two gradient buckets of the benchmark; "list": the four sizes of the
           small test bucket; "layers": T tensors with log-normal shares of N elements, as the layers of
           a network have; "flat": one tensor of N elements; "buckets": N elements in fixed-length
           buckets of d elements, each quantized on its own.
  scheme   "orq" (s = 3, 5, 9, 17 levels, unbiased), "bingrad_b", "bingrad_pb" (s = 2).
  values   distribution of the values of the "layers", "flat" and "buckets" layouts.
  clip     0, or c of the clipping to c standard deviations that goes before the quantizer.
  wire     "bits": bit-packed codes; "dense": base-s words (ORQ without clipping).
  iters    Lloyd updates (bingrad_b) or refinement sweeps (ORQ in fixed-length buckets).
  K        workers whose codes are summed (0 where nothing is decoded).
"""
import math
import random

import torch

import paper_2002_11082_b200 as ogq
from ogq_workloads import numel, resnet50_shapes, vgg19_shapes

SCHEMES = {"orq": ogq.OGQ_ORQ, "bingrad_b": ogq.OGQ_BINGRAD_B, "bingrad_pb": ogq.OGQ_BINGRAD_PB}
RESNET50, VGG19 = 25557032, 143667240  # elements of the two buckets


def _case(op, layout, scheme, s, N, T=1, d=0, K=0, values="laplace", clip=0.0, wire="bits", iters=0):
    return {"op": op, "layout": layout, "scheme": scheme, "s": s, "N": N, "T": T, "d": d, "K": K, "values": values,
            "clip": clip, "wire": wire, "iters": iters}


def listed():
    cases = {
        # the smallest use: one 256 KB gradient, 1-bit codes, encoded and decoded again (latency and launches)
        "flat64k_bingrad_b": _case("step", "flat", "bingrad_b", 2, 65536, K=1),
        # a small model's few tensors of unequal size and unlike distributions
        "list4_bingrad_pb": _case("encode", "list", "bingrad_pb", 2, 1380352, T=4),
        # a CNN's whole gradient, many small tensors among the large ones: the worker's side ...
        "resnet50_orq9": _case("encode", "resnet50", "orq", 9, RESNET50, T=161),
        # ... the same with the clipping of the ImageNet runs and ternary codes ...
        "resnet50_orq3_clip": _case("encode", "resnet50", "orq", 3, RESNET50, T=161, clip=2.5),
        # ... the server's side for eight workers ...
        "resnet50_orq9_decode": _case("decode", "resnet50", "orq", 9, RESNET50, T=161, K=8),
        # ... and the whole step in the entropy-dense wire format
        "resnet50_orq5_dense": _case("step", "resnet50", "orq", 5, RESNET50, T=161, K=8, wire="dense"),
        # a gradient that one fully connected weight dominates, in nine levels and in one bit
        "vgg19_orq9": _case("encode", "vgg19", "orq", 9, VGG19, T=38),
        "vgg19_bingrad_b": _case("encode", "vgg19", "bingrad_b", 2, VGG19, T=38),
        "vgg19_bingrad_b_decode": _case("decode", "vgg19", "bingrad_b", 2, VGG19, T=38, K=8),
        # one long vector of no round size, at the most levels
        "flat_odd_orq17": _case("encode", "flat", "orq", 17, 50000003, values="student_t4"),
        # fixed-length buckets: the ImageNet setting (d = 512, clipped), and the CIFAR one (d = 2048) as a whole step
        "buckets512_orq9_clip": _case("encode", "buckets", "orq", 9, RESNET50, T=49917, d=512, clip=2.5),
        "buckets2048_orq5": _case("step", "buckets", "orq", 5, 1700003, T=831, d=2048, K=4, values="student_t4"),
    }
    return [dict(c, name=name) for name, c in cases.items()]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: layers, a flat vector or fixed-length buckets, 4 K elements to the size of the VGG-19 bucket
    (fixed-length buckets: to that of ResNet-50)."""
    op = rng.choice(["encode", "encode", "decode", "step"])
    layout = rng.choice(["layers", "layers", "flat", "buckets", "buckets"])
    scheme = rng.choice(["orq", "orq", "orq", "bingrad_b", "bingrad_pb"])
    s = rng.choice([3, 5, 9, 17]) if scheme == "orq" else 2
    values = rng.choice(["laplace", "gaussian", "student_t4", "mixture"])
    clip = rng.choice([0.0, 0.0, 1.7, 2.5])
    wire = "dense" if scheme == "orq" and clip == 0.0 and layout != "buckets" and rng.random() < 0.25 else "bits"
    iters = rng.randint(1, 3) if rng.random() < 0.2 and (scheme == "bingrad_b" or (layout == "buckets" and scheme == "orq")) else 0
    K = _log(rng, 1, 16) if op != "encode" else 0
    top = RESNET50 if layout == "buckets" else VGG19
    # the codes of 16 workers of the largest bucket would cost more than any listed case; so would encode and decode of it
    N = _log(rng, 4096, top if op == "encode" else top // 2 if K <= 8 else top // 4)
    T, d = 1, 0
    if layout == "buckets":
        d = 128 << rng.randint(0, 8) if rng.random() < 0.75 else 128 * _log(rng, 1, 256)
        T = -(-N // d)
    elif layout == "layers":
        T = _log(rng, 2, min(200, N // 64))
    return _case(op, layout, scheme, s, N, T, d, K, values, clip, wire, iters)


# ------------------------------------------------------------------------------------------ inputs


def _sizes(case):
    """Element counts of the tensors (or buckets) of a case."""
    layout, N, T = case["layout"], case["N"], case["T"]
    if layout == "resnet50":
        return [numel(shape) for _, shape in resnet50_shapes()]
    if layout == "vgg19":
        return [numel(shape) for _, shape in vgg19_shapes()]
    if layout == "list":
        return [1 << 20, 1 << 18, 1 << 16, 1 << 12]
    if layout == "flat":
        return [N]
    if layout == "buckets":
        d = case["d"]
        return [d] * (N // d) + ([N % d] if N % d else [])
    rng = random.Random(N * 1000 + T)  # the architecture: the same for every seed of a case
    w = [math.exp(rng.gauss(0.0, 2.0)) for _ in range(T)]
    cut, acc, total = [0], 0.0, sum(w)
    for x in w:
        acc += x
        cut.append(min(N, int(N * acc / total)))
    cut[-1] = N
    return [b - a for a, b in zip(cut, cut[1:])]


def _distributions(case):
    layout = case["layout"]
    if layout == "resnet50":
        return ["laplace" if kind in ("conv", "fc_weight") else "gaussian" for kind, _ in resnet50_shapes()]
    if layout == "vgg19":
        return ["student_t4"] * case["T"]
    if layout == "list":
        return ["gaussian", "laplace", "student_t4", "mixture"]
    return [case["values"]] * (1 if layout in ("flat", "buckets") else case["T"])


def _fill(v, kind, gen):
    """Standard values of one distribution into v."""
    def u():
        return torch.rand(v.shape, device=v.device, generator=gen).clamp_(min=2.0 ** -25)

    if kind == "laplace":
        v.copy_(u()).log_().mul_(torch.where(u() < 0.5, 1.0, -1.0))
    elif kind == "gaussian":
        v.normal_(generator=gen)
    elif kind == "student_t4":  # z / sqrt(chi2_4 / 4), chi2_4 = -2 log(u1 u2)
        den = u().mul_(u()).log_().mul_(-0.5).clamp_(min=1e-12).sqrt_()
        v.normal_(generator=gen).div_(den)
    else:  # nine in ten from N(0, 1), the others from N(0, 100^2)
        v.normal_(generator=gen).mul_(torch.where(u() < 0.9, 1.0, 100.0))


def _gradient(case, sizes, gen):
    """A worker's gradient: every tensor with a scale of its own, 1e-5 to 1e-2, as the layers of a network have."""
    g = torch.empty(case["N"], device="cuda")
    kinds = _distributions(case)
    if len(kinds) == 1:
        _fill(g, kinds[0], gen)
        return g.mul_(1e-3)
    rng = random.Random(3)
    at = 0
    if len(set(kinds)) == 1:
        _fill(g, kinds[0], gen)
    for n, kind in zip(sizes, kinds):
        part = g[at:at + n]
        if len(set(kinds)) > 1:
            _fill(part, kind, gen)
        part.mul_(10.0 ** rng.uniform(-5.0, -2.0))
        at += n
    return g


class _Worker:
    """A worker's level tables and packed codes."""

    def __init__(self, T, s, words):
        self.levels = torch.zeros((T, s), device="cuda")
        self.thresh = torch.zeros(T, device="cuda")
        self.tau = torch.zeros(T, device="cuda")
        self.status = torch.zeros(T, dtype=torch.int32, device="cuda")
        self.packed = torch.zeros(words, dtype=torch.int32, device="cuda")


class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.case, st.seed = case, seed
    st.scheme = SCHEMES[case["scheme"]]
    s, N, T, d = case["s"], case["N"], case["T"], case["d"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    sizes = _sizes(case)
    if d:
        words = ogq.ogq_bucket_packed_words(N, d, ogq.ogq_bits_for_levels(s))
    else:
        h_off = [0]
        for n in sizes:
            h_off.append(h_off[-1] + n)
        h_po = ogq.ogq_dense_layout(h_off, s) if case["wire"] == "dense" else ogq.ogq_packed_layout(h_off, ogq.ogq_bits_for_levels(s))
        st.off, st.po, words = torch.tensor(h_off, device="cuda"), torch.from_numpy(h_po).cuda(), int(h_po[-1])
        st.ws_bytes = ogq.ogq_workspace_bytes(T, N, max(s, 3))
        st.ws = torch.empty(st.ws_bytes, dtype=torch.uint8, device="cuda")
    st.workers = [_Worker(T, s, words) for _ in range(max(1, case["K"]))]
    st.grad = None
    if case["op"] != "encode":  # the other workers' codes, as they were received
        st.packed_k = ogq.device_pointer_array([w.packed for w in st.workers])
        st.levels_k = ogq.device_pointer_array([w.levels for w in st.workers])
        st.out = torch.zeros(N, device="cuda")
        for k in range(len(st.workers)):
            st.grad = None
            st.grad = _gradient(case, sizes, gen)
            _encode(st, k)
    if case["op"] == "decode":
        torch.cuda.synchronize()
        st.grad = None
    else:
        st.grad = None
        st.grad = _gradient(case, sizes, gen)
    return st


# ------------------------------------------------------------------------------------------ one pass


def _encode(st, k):
    """Levels, quantize and pack of the gradient as worker k."""
    c, w = st.case, st.workers[k]
    s, N, T = c["s"], c["N"], c["T"]
    if c["d"]:
        ogq.ogq_bucket_encode(st.grad, N, c["d"], st.scheme, s, c["iters"], c["clip"], st.seed, k, w.levels, w.thresh, w.status, w.packed)
        return
    if c["clip"]:
        ogq.ogq_clip_threshold(st.grad, st.off, T, N, c["clip"], w.tau, w.status, st.ws, st.ws_bytes)
        if c["scheme"] == "orq":
            ogq.ogq_levels_orq_clipped(st.grad, st.off, T, N, s, w.tau, w.levels, w.status, st.ws, st.ws_bytes)
        else:
            ogq.ogq_levels_bingrad_clipped(st.grad, st.off, T, N, st.scheme, c["iters"], w.tau, w.levels, w.thresh, w.status, st.ws, st.ws_bytes)
        ogq.ogq_quantize_pack_clipped(st.grad, st.off, T, N, st.scheme, s, w.levels, w.thresh, w.tau, st.seed, k, st.po, w.packed)
        return
    if c["scheme"] == "orq":
        ogq.ogq_levels_orq(st.grad, st.off, T, N, s, w.levels, w.status, st.ws, st.ws_bytes)
    else:
        ogq.ogq_levels_bingrad(st.grad, st.off, T, N, st.scheme, c["iters"], w.levels, w.thresh, w.status, st.ws, st.ws_bytes)
    if c["wire"] == "dense":
        ogq.ogq_quantize_pack_dense(st.grad, st.off, T, N, s, w.levels, st.seed, k, st.po, w.packed)
    else:
        ogq.ogq_quantize_pack(st.grad, st.off, T, N, st.scheme, s, w.levels, w.thresh, st.seed, k, st.po, w.packed)


def _decode(st):
    c, K = st.case, st.case["K"]
    if c["d"]:
        ogq.ogq_bucket_decode_sum(st.packed_k, st.levels_k, K, c["N"], c["d"], c["s"], 1.0 / K, st.out)
    elif c["wire"] == "dense":
        ogq.ogq_unpack_sum_dense(st.packed_k, st.levels_k, K, st.off, st.po, c["T"], c["N"], c["s"], 1.0 / K, st.out)
    else:
        ogq.ogq_unpack_sum(st.packed_k, st.levels_k, K, st.off, st.po, c["T"], c["N"], c["s"], 1.0 / K, st.out)


def run(st):
    op, got = st.case["op"], {}
    if op != "decode":
        _encode(st, 0)
        w = st.workers[0]
        got.update(levels=w.levels, status=w.status, packed=w.packed)
        if st.case["scheme"] == "bingrad_b":
            got["thresh"] = w.thresh
        if st.case["clip"] and not st.case["d"]:
            got["tau"] = w.tau
    if op != "encode":
        _decode(st)
        got["out"] = st.out
    return got


def work(case):
    """The gradient read once and its codes and levels written once; the K workers' codes and levels read once and their
    sum written once.  The operations are neither matrix work nor what bounds the path."""
    s, N, T, K = case["s"], case["N"], case["T"], case["K"]
    codes = N * (32.0 / ogq.ogq_dense_digits(s) if case["wire"] == "dense" else ogq.ogq_bits_for_levels(s)) / 8.0
    level_bytes = 4.0 * T * s
    total = 0.0
    if case["op"] != "decode":
        total += 4.0 * N + codes + level_bytes
    if case["op"] != "encode":
        total += K * (codes + level_bytes) + 4.0 * N
        if case["op"] == "step":
            total -= codes + level_bytes  # the own codes need not be read back
    return {"bytes": total, "flops": 0.0}


def tolerance(case):
    """ORQ levels are values of the data and codes follow from levels and counter-based random numbers; means, standard
    deviations and the BinGrad-pb level are fp64 sums rounded to fp32, where another order of summation can move the last
    bit, and with it one code in some 10^7.  The sums are of up to 16 fp32 terms in a fixed order."""
    return {"rel": 1e-6, "max": 1e-5, "differ": 1e-5}

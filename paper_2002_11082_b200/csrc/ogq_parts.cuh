// Tensor-wise sums over the flat bucket, as BinGrad-b and the clipping threshold take them: pieces of the
// tensors larger than kSoloN are summed by flat CTAs into fixed slots, which a CTA per tensor adds up in CTA
// order in the next launch; smaller tensors belong to one CTA from start to finish.
//
// (The combination used to be done by the last CTA to arrive for a tensor, with a counter to clear before
// and a fence and an atomic per piece; and a chunk full of tiny tensors went through that for each of
// them, 3 to 4 us a piece, while the other CTAs had long finished.)
#pragma once

#include "ogq_common.cuh"
#include "ogq_ws.h"

namespace ogq {

constexpr int kSoloN = 16384;

// Where a flat CTA leaves the partial sums of its piece of tensor t.
__device__ __forceinline__ BbPart* part_slot(const BbWs& ws, int t, int64_t tb, int64_t te, int64_t chunk)
{
    const int64_t c = blockIdx.x, lo = c * chunk;
    if (tb / chunk == (te - 1) / chunk) return ws.direct + t;
    return tb < lo ? ws.slot_a + c : ws.slot_b + c;
}

struct PartSum {
    double s_lo, s_hi;
    long long c_lo, c_hi;
};

// All partial sums of tensor t, in CTA order: called by all threads of a CTA, valid in thread 0.
__device__ __forceinline__ PartSum part_total(const BbWs& ws, int t, int64_t tb, int64_t te, int64_t chunk, double* sh_d,
                                              long long* sh_l)
{
    const int64_t c0 = tb / chunk, c1 = (te - 1) / chunk;
    PartSum r = {0.0, 0.0, 0, 0};
    for (int64_t c = c0 + threadIdx.x; c <= c1; c += kThreads) {
        const BbPart* p = c0 == c1 ? ws.direct + t : (c == c0 ? ws.slot_b + c : ws.slot_a + c);
        r.s_lo += __ldcg(&p->s_lo);
        r.s_hi += __ldcg(&p->s_hi);
        r.c_lo += __ldcg(&p->c_lo);
        r.c_hi += __ldcg(&p->c_hi);
    }
    r.s_lo = block_sum(r.s_lo, sh_d);
    r.s_hi = block_sum(r.s_hi, sh_d);
    r.c_lo = block_sum(r.c_lo, sh_l);
    r.c_hi = block_sum(r.c_hi, sh_l);
    return r;
}

}  // namespace ogq

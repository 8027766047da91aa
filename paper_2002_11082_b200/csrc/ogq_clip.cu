// Gradient clipping threshold: tau = c * sigma per tensor, sigma^2 the variance of the tensor about
// its mean (Section "Experiments", paragraph after the list of methods: clip(v) = sign(v) min(|v|, c sigma)).
//
// One streaming read.  Sums of (v - v0) and (v - v0)^2 with v0 the tensor's first element are
// accumulated in fp64 per thread and combined in a fixed order (per-CTA slots, added up in CTA order by a
// CTA per tensor in the next launch; tensors of up to kSoloN elements by the one CTA that reads them); the
// variance is (S2 - S1^2 / n) / n, which the shift by v0 keeps free of the cancellation a large mean would
// cause.  The clamp itself is applied by the level solvers as they read the gradient (the clipped gradient
// is never written out).
#include <math.h>

#include "ogq_common.cuh"
#include "ogq_internal.h"
#include "ogq_parts.cuh"
#include "ogq_ws.h"

namespace ogq {

struct ClipArgs {
    const float* grad;
    const int64_t* off;
    int T;
    int64_t total, chunk;
    float c;
    float* tau;
    int32_t* status;
    BbWs ws;
};

// S1 in s_lo, S2 in s_hi, whether a value is not finite in c_lo; valid in thread 0.
__device__ __forceinline__ PartSum clip_sums(const float* __restrict__ grad, int64_t tb, int64_t pb, int64_t pe, double* sh_d)
{
    const double v0 = (double)__ldg(grad + tb);
    // two accumulators for each sum, taken in turn: the chain of dependent additions is what a thread waits for
    double a1 = 0.0, b1 = 0.0, a2 = 0.0, b2 = 0.0;
    uint32_t top = 0u;
    visit_piece(grad, pb, pe, [&](float v) {
        top = max(top, __float_as_uint(v) & 0x7fffffffu);
        const double d = (double)v - v0;
        const double n1 = a1 + d, n2 = a2 + d * d;
        a1 = b1; b1 = n1;
        a2 = b2; b2 = n2;
    });
    PartSum r;
    r.s_lo = block_sum(a1 + b1, sh_d);
    r.s_hi = block_sum(a2 + b2, sh_d);
    r.c_lo = __syncthreads_or(top >= 0x7f800000u) ? 1 : 0;
    r.c_hi = 0;
    return r;
}

__device__ __forceinline__ void clip_finish(const ClipArgs& A, int t, const PartSum& a, int64_t n)
{
    if (a.c_lo) {
        A.tau[t] = 0.f;
        A.status[t] = OGQ_ST_NONFINITE;
        return;
    }
    double var = (a.s_hi - a.s_lo * a.s_lo / (double)n) / (double)n;
    if (!(var > 0.0)) var = 0.0;
    A.tau[t] = (float)((double)A.c * sqrt(var));
    A.status[t] = 0;
}

// Grid: the flat CTAs, then one CTA per tensor for the tensors of up to kSoloN elements.
__global__ void __launch_bounds__(kThreads) k_clip_threshold(ClipArgs A, int flat_ctas)
{
    __shared__ double sh_d[kWarps];
    pdl_wait();
    pdl_launch_dependents();
    if ((int)blockIdx.x >= flat_ctas) {
        const int t = blockIdx.x - flat_ctas;
        const int64_t tb = __ldg(A.off + t), te = __ldg(A.off + t + 1);
        if (te - tb > kSoloN) return;
        if (te <= tb) {
            if (threadIdx.x == 0) {
                A.tau[t] = 0.f;
                A.status[t] = OGQ_ST_EMPTY;
            }
            return;
        }
        const PartSum a = clip_sums(A.grad, tb, tb, te, sh_d);
        if (threadIdx.x == 0) clip_finish(A, t, a, te - tb);
        return;
    }
    const int64_t lo = (int64_t)blockIdx.x * A.chunk;
    const int64_t hi = (lo + A.chunk < A.total) ? lo + A.chunk : A.total;
    for_each_piece(A.off, A.T, lo, hi, [&](int t, int64_t tb, int64_t te, int64_t pb, int64_t pe) {
        if (te - tb <= kSoloN) return;
        const PartSum a = clip_sums(A.grad, tb, pb, pe, sh_d);
        if (threadIdx.x == 0) {
            BbPart p;
            p.s_lo = a.s_lo; p.s_hi = a.s_hi; p.c_lo = a.c_lo; p.c_hi = 0;
            *part_slot(A.ws, t, tb, te, A.chunk) = p;
        }
    });
}

// One CTA per tensor: adds up the partial sums.
__global__ void __launch_bounds__(kThreads) k_clip_combine(ClipArgs A)
{
    __shared__ double sh_d[kWarps];
    __shared__ long long sh_l[kWarps];
    pdl_wait();
    pdl_launch_dependents();
    const int t = blockIdx.x;
    const int64_t tb = __ldg(A.off + t), te = __ldg(A.off + t + 1);
    if (te - tb <= kSoloN) return;
    const PartSum a = part_total(A.ws, t, tb, te, A.chunk, sh_d, sh_l);
    if (threadIdx.x == 0) clip_finish(A, t, a, te - tb);
}

cudaError_t launch_clip_threshold(const float* d_grad, const int64_t* d_off, int T, int64_t total, float c,
                                  float* d_tau, int32_t* d_status, void* d_ws, int sm_count, cudaStream_t stream)
{
    const FlatGrid g = make_flat_grid(total, sm_count * 4 < kMaxFlatCtas ? sm_count * 4 : kMaxFlatCtas, 8192);
    ClipArgs A;
    A.grad = d_grad; A.off = d_off; A.T = T; A.total = total; A.chunk = g.chunk; A.c = c; A.tau = d_tau; A.status = d_status;
    A.ws = bb_ws_carve(d_ws, T, g.ctas);
    const int flat = total > kSoloN ? g.ctas : 0;  // some tensor may be larger than one CTA takes on its own
    launch_begin("k_clip_threshold", stream);
    cudaError_t e = launch_pdl(k_clip_threshold, flat + T, kThreads, 0, stream, A, flat);
    launch_end(stream);
    if (flat == 0 || e != cudaSuccess) return e;
    launch_begin("k_clip_combine", stream);
    e = launch_pdl(k_clip_combine, T, kThreads, 0, stream, A);
    launch_end(stream);
    return e;
}

}  // namespace ogq

// BinGrad-b level solver: Eq. (bingrad-b optimal condition).
//
// Pass 0 streams the bucket once for the per-tensor sum (b_0 = mean).  Every
// further pass streams it again for the counts and sums of {v < b_0} and
// {v >= b_0}, i.e. the two conditional means; with Lloyd iterations requested
// the launch that adds a pass's partial sums up moves b_0 to the midpoint and
// the next pass repeats.  Partial sums are fp64, written to fixed slots and
// combined in CTA order, so results do not depend on scheduling.  Tensors of up
// to kSoloN elements are solved by a CTA of their own in the first launch.
#include <math.h>

#include <atomic>

#include "ogq_common.cuh"
#include "ogq_internal.h"
#include "ogq_parts.cuh"
#include "ogq_ws.h"

namespace ogq {

struct BbArgs {
    const float* grad;
    const int64_t* off;
    int T;
    int64_t total, chunk;
    int lloyd_iters;
    const float* tau;
    float* levels;
    float* thresh;
    int32_t* status;
    BbWs ws;
};

// Sums of {v < b0} and {v >= b0} of grad[pb, pe) over the CTA; valid in thread 0.  CLIP: every value is first
// clamped to [-tau, tau].
template <bool CLIP, bool WIDE = false>
__device__ __forceinline__ PartSum bb_split(const float* __restrict__ grad, int64_t pb, int64_t pe, float b0, float tau,
                                            double* sh_d, long long* sh_l, bool down = false)
{
    PartSum r = {0.0, 0.0, 0, 0};
    int below = 0;
    auto add = [&](float raw) {
        const float v = CLIP ? copysignf(fminf(fabsf(raw), tau), raw) : raw;
        const bool b = v < b0;
        const double d = (double)v;
        r.s_lo += b ? d : 0.0;
        r.s_hi += b ? 0.0 : d;
        below += b ? 1 : 0;
    };
    if constexpr (WIDE) visit_piece_wide(grad, pb, pe, add, down);
    else visit_piece(grad, pb, pe, add, down);
    r.s_lo = block_sum(r.s_lo, sh_d);
    r.s_hi = block_sum(r.s_hi, sh_d);
    r.c_lo = block_sum((long long)below, sh_l);
    r.c_hi = (pe - pb) - r.c_lo;
    return r;
}

// What a complete pass says about a tensor: pass 0 gives b_0, every later one the levels and, while Lloyd
// updates are left, the next b_0.  Returns true when the tensor is finished.
struct BbState {
    float b0, l_lo, l_hi;
    int status;
    long long prev_lo;
};

__device__ __forceinline__ bool bb_advance(const PartSum& a, int pass, int lloyd_iters, BbState& st)
{
    if (pass == 0) {
        st.status = isfinite(a.s_hi) ? 0 : OGQ_ST_NONFINITE;
        st.b0 = (float)(a.s_hi / (double)a.c_hi);
        st.prev_lo = -1;
        return false;
    }
    if (a.c_lo == 0 || a.c_hi == 0) {
        const double m = (a.c_lo == 0) ? a.s_hi / (double)a.c_hi : a.s_lo / (double)a.c_lo;
        st.l_lo = st.l_hi = (float)m;
        st.status |= OGQ_ST_CONSTANT;
        return true;
    }
    const double m_lo = a.s_lo / (double)a.c_lo, m_hi = a.s_hi / (double)a.c_hi;
    st.l_lo = (float)m_lo;
    st.l_hi = (float)m_hi;
    if (a.c_lo == st.prev_lo) return true;
    if (pass - 1 >= lloyd_iters) {
        if (lloyd_iters > 0) st.status |= OGQ_ST_ITER_CAP;
        return true;
    }
    st.prev_lo = a.c_lo;
    st.b0 = (float)((m_lo + m_hi) * 0.5);
    return false;
}

// Barrier of the cluster's CTAs; shared-memory writes before it are seen after it.
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// *p in the shared memory of the cluster's CTA `rank` (p: the address in this CTA's own).
__device__ __forceinline__ PartSum cluster_load(const PartSum* p, int rank)
{
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm("mapa.shared::cluster.u32 %0, %0, %1;" : "+r"(a) : "r"(rank));
    PartSum r;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(r.s_lo) : "r"(a));
    asm volatile("ld.shared::cluster.f64 %0, [%1+8];" : "=d"(r.s_hi) : "r"(a));
    asm volatile("ld.shared::cluster.s64 %0, [%1+16];" : "=l"(r.c_lo) : "r"(a));
    asm volatile("ld.shared::cluster.s64 %0, [%1+24];" : "=l"(r.c_hi) : "r"(a));
    return r;
}

// Grid: the flat CTAs, and in pass 0 after them one CTA per tensor for the tensors of up to kSoloN elements.
//   Pass bound: DRAM where the bucket exceeds L2 (143.7 M elements: 92 us, 6.2 TB/s); small buckets: the
// latency of one load and one block sum.
//   48 registers: an SM takes a fifth CTA beside the grid's four.  With 62 the passes of eight workers on eight streams had no room
// for one another (ResNet-50 bucket: 411 us, now 377), and neither had the CTAs of small tensors (9000 of 3000 elements: 148, now
// 139).  The clipped passes, which wait for fp64 as much as for DRAM, had 60 before the wide loads and keep 64.
template <bool CLIP>
__global__ void __launch_bounds__(kThreads, CLIP ? 4 : 5) k_bb_pass(BbArgs A, int flat_ctas, int pass)
{
    __shared__ double sh_d[kWarps];
    __shared__ long long sh_l[kWarps];
    __shared__ float sh_b0;
    pdl_wait();
    pdl_launch_dependents();

    if ((int)blockIdx.x >= flat_ctas) {
        const int t = blockIdx.x - flat_ctas;
        const int64_t tb = __ldg(A.off + t), te = __ldg(A.off + t + 1);
        if (te - tb > kSoloN) return;
        if (te <= tb) {
            if (threadIdx.x == 0) {
                A.levels[2 * t] = 0.f;
                A.levels[2 * t + 1] = 0.f;
                A.thresh[t] = 0.f;
                A.status[t] = OGQ_ST_EMPTY;
            }
            return;
        }
        const float tau = CLIP ? __ldcg(A.tau + t) : 0.f;
        BbState st;
        float b0 = -INFINITY;
        for (int p = 0;; ++p) {
            const PartSum a = bb_split<CLIP, true>(A.grad, tb, te, b0, tau, sh_d, sh_l);
            bool end = false;
            if (threadIdx.x == 0) {
                end = bb_advance(a, p, A.lloyd_iters, st);
                sh_b0 = st.b0;
            }
            end = __syncthreads_or(end);
            if (end) break;
            b0 = sh_b0;
        }
        if (threadIdx.x == 0) {
            A.levels[2 * t] = st.l_lo;
            A.levels[2 * t + 1] = st.l_hi;
            A.thresh[t] = st.b0;
            A.status[t] = st.status;
        }
        return;
    }

    const int64_t lo = (int64_t)blockIdx.x * A.chunk;
    const int64_t hi = (lo + A.chunk < A.total) ? lo + A.chunk : A.total;
    const bool down = ((pass & 1) != 0) != CLIP;  // the passes go up and down in turn, after the clipping threshold's upward one
    for_each_piece(A.off, A.T, lo, hi, [&](int t, int64_t tb, int64_t te, int64_t pb, int64_t pe) {
        if (te - tb <= kSoloN || (pass > 0 && __ldcg(A.ws.done + t))) return;
        const float b0 = pass == 0 ? -INFINITY : __ldcg(A.thresh + t);
        const PartSum a = bb_split<CLIP, true>(A.grad, pb, pe, b0, CLIP ? __ldcg(A.tau + t) : 0.f, sh_d, sh_l, down);
        if (threadIdx.x == 0) {
            BbPart p;
            p.s_lo = a.s_lo; p.s_hi = a.s_hi; p.c_lo = a.c_lo; p.c_hi = a.c_hi;
            *part_slot(A.ws, t, tb, te, A.chunk) = p;
        }
    }, down);
}

// One CTA per tensor: adds up the partial sums of the pass before.
__global__ void __launch_bounds__(kThreads) k_bb_combine(BbArgs A, int pass)
{
    __shared__ double sh_d[kWarps];
    __shared__ long long sh_l[kWarps];
    pdl_wait();
    pdl_launch_dependents();
    const int t = blockIdx.x;
    const int64_t tb = __ldg(A.off + t), te = __ldg(A.off + t + 1);
    if (te - tb <= kSoloN || (pass > 0 && __ldcg(A.ws.done + t))) return;
    const PartSum a = part_total(A.ws, t, tb, te, A.chunk, sh_d, sh_l);
    if (threadIdx.x == 0) {
        BbState st = {0.f, 0.f, 0.f, 0, -1};
        if (pass > 0) {
            st.b0 = __ldcg(A.thresh + t);
            st.status = __ldcg(A.status + t);
            st.prev_lo = __ldcg(A.ws.prev_lo + t);
        }
        const bool end = bb_advance(a, pass, A.lloyd_iters, st);
        if (pass > 0) {
            A.levels[2 * t] = st.l_lo;
            A.levels[2 * t + 1] = st.l_hi;
        }
        A.thresh[t] = st.b0;
        A.status[t] = st.status;
        A.ws.prev_lo[t] = st.prev_lo;
        A.ws.done[t] = end ? 1 : 0;
    }
}

// Small buckets: a cluster of kBbCluster CTAs per tensor does all passes in one launch, the partial sums meet
// in the CTAs' shared memory.  A bucket of up to kBbClusterN elements is a matter of latencies: one launch
// of 6 us instead of two passes and two combinations (4 launches, 12 us, and 12 us of host time).  Above, a
// CTA's share takes longer than the launches it saves.
constexpr int kBbCluster = 8;
constexpr int kBbClusterN = 131072, kBbClusterT = 128;

template <bool CLIP>
__global__ void __cluster_dims__(kBbCluster, 1, 1) __launch_bounds__(kThreads) k_bb_cluster(BbArgs A)
{
    __shared__ double sh_d[kWarps];
    __shared__ long long sh_l[kWarps];
    __shared__ PartSum sh_part[2];  // this CTA's sums of the even and the odd passes
    pdl_wait();
    pdl_launch_dependents();
    const int t = blockIdx.x / kBbCluster, rank = blockIdx.x % kBbCluster;
    const int64_t tb = __ldg(A.off + t), te = __ldg(A.off + t + 1), n = te - tb;
    if (n <= 0) {
        if (rank == 0 && threadIdx.x == 0) {
            A.levels[2 * t] = 0.f;
            A.levels[2 * t + 1] = 0.f;
            A.thresh[t] = 0.f;
            A.status[t] = OGQ_ST_EMPTY;
        }
        return;  // the whole cluster
    }
    const int64_t share = ((n + kBbCluster - 1) / kBbCluster + 3) & ~(int64_t)3;
    int64_t pb = tb + rank * share, pe = pb + share;
    if (pb > te) pb = te;
    if (pe > te) pe = te;
    const float tau = CLIP ? __ldcg(A.tau + t) : 0.f;
    BbState st;
    st.b0 = -INFINITY;
    for (int p = 0;; ++p) {
        const PartSum mine = bb_split<CLIP>(A.grad, pb, pe, st.b0, tau, sh_d, sh_l);
        if (threadIdx.x == 0) sh_part[p & 1] = mine;
        cluster_sync();
        // every thread of every CTA adds the shares up in rank order and so takes the same decision; the sums of
        // the next pass go to the other slot, so one barrier per pass is enough
        PartSum a = {0.0, 0.0, 0, 0};
#pragma unroll
        for (int r = 0; r < kBbCluster; ++r) {
            const PartSum q = cluster_load(&sh_part[p & 1], r);
            a.s_lo += q.s_lo; a.s_hi += q.s_hi; a.c_lo += q.c_lo; a.c_hi += q.c_hi;
        }
        if (bb_advance(a, p, A.lloyd_iters, st)) break;
    }
    if (rank == 0 && threadIdx.x == 0) {
        A.levels[2 * t] = st.l_lo;
        A.levels[2 * t + 1] = st.l_hi;
        A.thresh[t] = st.b0;
        A.status[t] = st.status;
    }
    cluster_sync();  // a CTA's shared memory stays until the others have read it
}

// From this size on a pass keeps the fifth place of every SM empty, with shared memory that it does not use.  A pass is launched
// while the kernel before it drains; SMs that are done early otherwise take five of its CTAs and others three, and the whole
// waits for the SMs with five (one worker, encode: 143.7 M elements 298 and 280 us, 40 M 89 and 86).  Smaller buckets lose
// less by it than several streams gain (ResNet-50 bucket, eight streams: 378 us, 409 with the place kept empty; one stream:
// 67 us either way behind a threshold quantizer that lets a pass be launched late, see there).
constexpr int64_t kBbAloneN = 32 << 20;
constexpr size_t kBbAloneBytes = 46 * 1024;  // four CTAs fit an SM, five do not

static FlatGrid bb_grid(int64_t total, int sm_count)
{
    return make_flat_grid(total, sm_count * 4 < kMaxFlatCtas ? sm_count * 4 : kMaxFlatCtas, 8192);
}

static cudaError_t bb_run(const float* d_grad, const int64_t* d_off, int T, int64_t total, const FlatGrid& g, int lloyd_iters,
                          const float* d_tau, float* d_levels, float* d_thresh, int32_t* d_status, void* scratch,
                          cudaStream_t stream)
{
    BbArgs A;
    A.grad = d_grad; A.off = d_off; A.T = T; A.total = total; A.chunk = g.chunk; A.lloyd_iters = lloyd_iters; A.tau = d_tau;
    A.levels = d_levels; A.thresh = d_thresh; A.status = d_status; A.ws = bb_ws_carve(scratch, T, g.ctas);
    if (total <= kBbClusterN && T <= kBbClusterT) {
        launch_begin("k_bb_cluster", stream);
        const cudaError_t e = launch_pdl(d_tau ? k_bb_cluster<true> : k_bb_cluster<false>, T * kBbCluster, kThreads, 0, stream, A);
        launch_end(stream);
        return e;
    }
    const int flat = total > kSoloN ? g.ctas : 0;  // some tensor may be larger than one CTA solves on its own
    auto kernel = d_tau ? k_bb_pass<true> : k_bb_pass<false>;
    const size_t unused = total >= kBbAloneN && T <= g.ctas ? kBbAloneBytes : 0;  // (not where CTAs of small tensors want the place)
    cudaError_t e = cudaSuccess;
    for (int pass = 0; pass <= lloyd_iters + 1 && e == cudaSuccess; ++pass) {
        launch_begin("k_bb_pass", stream);
        e = launch_pdl(kernel, flat + (pass == 0 ? T : 0), kThreads, unused, stream, A, flat, pass);
        launch_end(stream);
        if (flat == 0 || e != cudaSuccess) break;
        launch_begin("k_bb_combine", stream);
        e = launch_pdl(k_bb_combine, T, kThreads, 0, stream, A, pass);
        launch_end(stream);
    }
    return e;
}

cudaError_t launch_levels_bingrad_b(const float* d_grad, const int64_t* d_off, int T, int64_t total,
                                    int lloyd_iters, const float* d_tau, float* d_levels, float* d_thresh,
                                    int32_t* d_status, void* d_ws, int sm_count, cudaStream_t stream)
{
    return bb_run(d_grad, d_off, T, total, bb_grid(total, sm_count), lloyd_iters, d_tau, d_levels, d_thresh, d_status, d_ws,
                  stream);
}

size_t ws_bytes_bingrad_b(int T, int64_t /*total*/) { return bb_ws_bytes(T, kMaxFlatCtas); }

// ---------------------------------------------------------------------------
// Variant for callers that cannot allocate device memory: the scratch of the
// BinGrad-b solver lives in a fixed array inside the library image.  The array
// is sized for kNoAllocMaxTensors tensors and the largest flat grid; every GPU
// that loads the library keeps these ~304 KB until the process exits.
// ---------------------------------------------------------------------------
constexpr size_t kNoAllocBytes = 2 * ((sizeof(BbPart) * kMaxFlatCtas + 255) / 256 * 256) +
                                 (sizeof(BbPart) * kNoAllocMaxTensors + 255) / 256 * 256 +
                                 (sizeof(int) * kNoAllocMaxTensors + 255) / 256 * 256 +
                                 (sizeof(long long) * kNoAllocMaxTensors + 255) / 256 * 256;

static __device__ __align__(256) unsigned char g_bb_static_scratch[kNoAllocBytes];

// Device address of the array above, looked up once per device.  In host code the symbol's name is
// only a handle, not an address the GPU can use, so the address has to come from the runtime.
// Two host threads that make the first call on a device at the same time both look the address up and
// store the same value: the slot is atomic so that this is well defined.
static std::atomic<void*> g_bb_static_ptr[kNoAllocMaxDevices];

cudaError_t launch_levels_bingrad_b_static(const float* d_grad, const int64_t* d_off, int T, int64_t total,
                                           int lloyd_iters, float* d_levels, float* d_thresh,
                                           int32_t* d_status, int sm_count, cudaStream_t stream)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kNoAllocMaxDevices) return cudaErrorInvalidDevice;
    void* scratch = g_bb_static_ptr[dev].load(std::memory_order_acquire);
    if (scratch == nullptr) {
        e = cudaGetSymbolAddress(&scratch, g_bb_static_scratch);
        if (e != cudaSuccess) return e;
        g_bb_static_ptr[dev].store(scratch, std::memory_order_release);
    }
    const FlatGrid g = bb_grid(total, sm_count);
    // cannot happen for T <= kNoAllocMaxTensors (the caller checked): the array is sized for that many
    // tensors and the largest grid
    if (bb_ws_bytes(T, g.ctas) > kNoAllocBytes) return cudaErrorUnknown;
    return bb_run(d_grad, d_off, T, total, g, lloyd_iters, nullptr, d_levels, d_thresh, d_status, scratch, stream);
}

}  // namespace ogq

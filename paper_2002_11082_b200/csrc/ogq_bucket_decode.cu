// Server step of fixed-length buckets (the encoder is ogq_bucket.cu).
#include <type_traits>

#include "ogq_common.cuh"
#include "ogq_internal.h"
#include "ogq_quant.cuh"
#include "ogq_unpack.cuh"

namespace ogq {

// Server step for fixed-length buckets: out[i] = scale * sum_k levels_k[i / d][code_k[i]].  Because d is
// a multiple of 128, the packed codes of consecutive buckets form one contiguous bit stream (only the
// last, shorter bucket is padded).  A warp takes a run of consecutive groups of 256 elements, eight per lane, and keeps the
// workers' level rows of the group's one or two buckets (two: lanes 16 ... 31 are in the second) in shared
// memory until the bucket changes.  Same additions in the same (worker) order as ogq_unpack_sum with offsets j * d.
// PAIRS: two groups of one bucket at a time, twice the loads and reads in flight.
template <int BITS, int REST, bool PAIRS>
__global__ void __launch_bounds__(kThreads, 4)
k_bucket_decode_sum(const uint32_t* const* __restrict__ packed_k, const float* const* __restrict__ levels_k, int K,
                    int64_t total, int d, int nb, int s, int64_t total_words, float scale, float* __restrict__ outp)
{
    extern __shared__ __align__(256) unsigned char sh_rows[];  // [kWarps][2][row_bytes(K)]
    __shared__ const uint32_t* sh_pk[kMaxWorkers];
    __shared__ const float* sh_lp[kMaxWorkers];
    constexpr int R = kRowStride<BITS>, kWords = 8 * BITS;
    pdl_wait();
    pdl_launch_dependents();
    for (int k = threadIdx.x; k < K; k += kThreads) { sh_pk[k] = packed_k[k]; sh_lp[k] = levels_k[k]; }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t ngroups = (total + 255) >> 8, full = total >> 8;
    const int64_t nw = (int64_t)gridDim.x * kWarps, me = (int64_t)blockIdx.x * kWarps + warp;
    const int64_t g_beg = me * ngroups / nw, g_end = (me + 1) * ngroups / nw;
    if (g_beg >= g_end) return;
    const uint32_t rb = row_bytes<BITS>(K);
    unsigned char* rows = sh_rows + (size_t)warp * 2 * rb;
    const uint32_t rows_at = (uint32_t)__cvta_generic_to_shared(rows);
    const int shift = (int)((reinterpret_cast<uintptr_t>(outp) >> 2) & 3);
    int j = (int)((g_beg << 8) / d), at = (int)((g_beg << 8) - (int64_t)j * d);  // bucket of the group, first element in it
    int j_rows = -1, two_rows = 0;                                               // buckets the rows are of
    for (int64_t g = g_beg; g < g_end; ++g) {
        const int two = at + 128 >= d && j + 1 < nb;
        if (j != j_rows || two > two_rows) {
            __syncwarp();
            for (int i = lane; i < (K * R << two); i += 32) {
                const int q = i % R, kk = i / R, second = kk >= K;
                const int k = second ? kk - K : kk;
                reinterpret_cast<float*>(rows + (second ? rb : 0u))[k * R + q] = __ldcg(sh_lp[k] + (int64_t)(j + second) * s + (q < s ? q : s - 1));
            }
            __syncwarp();
            j_rows = j; two_rows = two;
        }
        const uint32_t other = two && lane >= 16 ? rb : 0u;
        const int64_t w0 = g * kWords;
        auto write = [&](int64_t q, float (&a)[8]) {
#pragma unroll
            for (int e = 0; e < 8; ++e) a[e] = __fmul_rn(a[e], scale);
            // (256-bit stores for 1-bit codes, too, with two groups at a time: there two 128-bit ones, which write every sector by halves, cost
            // 31.4 instead of 22.0 us for 25 M elements of one worker at d = 2048.  With one group at a time they are the
            // faster: 1.7 M elements of sixteen workers 9.1 instead of 9.7.)
            store8<(BITS > 1 || PAIRS)>(outp + (q << 8) + 8 * lane, shift, lane, a);
        };
        if (PAIRS && at + 512 <= d && g + 1 < g_end && g + 1 < full) {  // two groups of one bucket
            float a[2][8];
            sum_workers<BITS, 2, false, REST>(K, lane, 0u, rows_at, [&](int k, int q) { return sh_pk[k] + w0 + q * kWords; }, a);
            write(g, a[0]);
            write(g + 1, a[1]);
            ++g;
            at += 256;
        } else if (g < full) {
            float a[1][8];
            sum_workers<BITS, 1, false, REST>(K, lane, 0u, rows_at + other, [&](int k, int) { return sh_pk[k] + w0; }, a);
            write(g, a[0]);
        } else {  // the last, partial group
            const int64_t i0 = (g << 8) + 8 * lane, wi = (i0 * BITS) >> 5;
            if (i0 < total) {
                const int sh = (int)(i0 * BITS) & 31;
                const bool more = sh + 8 * BITS > 32 && wi + 1 < total_words;
                const float* mine = reinterpret_cast<const float*>(rows + other);
                float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                for (int k = 0; k < K; ++k) {
                    const uint32_t lo = __ldcg(sh_pk[k] + wi), hi = more ? __ldcg(sh_pk[k] + wi + 1) : 0u;
                    const uint64_t codes = ((uint64_t)hi << 32 | lo) >> sh;
#pragma unroll
                    for (int e = 0; e < 8; ++e) a[e] = __fadd_rn(a[e], mine[k * R + ((int)(codes >> (e * BITS)) & (R - 1))]);
                }
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (i0 + e < total) outp[i0 + e] = __fmul_rn(a[e], scale);
            }
        }
        for (at += 256; at >= d; at -= d) ++j;
    }
}

cudaError_t launch_bucket_decode_sum(const uint32_t* const* d_packed_k, const float* const* d_levels_k, int K,
                                     int64_t total, int d, int s, float scale, float* d_out, int sm_count,
                                     cudaStream_t stream)
{
    const int bits = ogq_bits_for_levels(s);
    const int64_t nb = (total + d - 1) / d;
    const int64_t last = total - (nb - 1) * d;
    const int64_t total_words = (nb - 1) * ((int64_t)d * bits / 32) + ((last * bits + 31) / 32 + 3) / 4 * 4;
    const int64_t ngroups = (total + 255) >> 8;
    int64_t ctas = (ngroups + kWarps - 1) / kWarps;
    if (ctas > (int64_t)sm_count * 4) ctas = (int64_t)sm_count * 4;
    size_t rows = 0;
    cudaError_t e = cudaSuccess;
    launch_begin("k_bucket_decode_sum", stream);
    // Two groups at a time in longer runs (20 M elements at d = 512, five workers of nine levels: 42.2 -> 35.3 us; d = 2048, six
    // of five levels: 44.4 -> 38.1); short runs spend more on fetching the instructions than it saves (5 M elements at d = 1024, ten
    // workers: 0.6 us longer).
    const bool pairs = ngroups >= ctas * kWarps * 8 && d >= 512;
#define OGQ_LAUNCH_BD(B)                                                                                        \
    do {                                                                                                        \
        rows = (size_t)kWarps * 2 * row_bytes<B>(K);                                                            \
        e = with_rest<B, false>(rest_of<B, false>(K), [&](auto rest) -> cudaError_t {                                  \
            auto kernel = pairs ? k_bucket_decode_sum<B, decltype(rest)::value, true>                           \
                                : k_bucket_decode_sum<B, decltype(rest)::value, false>;                         \
            if (rows > 40 * 1024) {                                                                             \
                const cudaError_t a = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024); \
                if (a != cudaSuccess) return a;                                                                 \
            }                                                                                                   \
            return launch_pdl(kernel, (int)ctas, kThreads, rows, stream, d_packed_k, d_levels_k, K, total, d,   \
                              (int)nb, s, total_words, scale, d_out);                                           \
        });                                                                                                     \
    } while (0)
    switch (bits) {
        case 1: OGQ_LAUNCH_BD(1); break;
        case 2: OGQ_LAUNCH_BD(2); break;
        case 3: OGQ_LAUNCH_BD(3); break;
        case 4: OGQ_LAUNCH_BD(4); break;
        case 5: OGQ_LAUNCH_BD(5); break;
        default: return cudaErrorInvalidValue;
    }
#undef OGQ_LAUNCH_BD
    launch_end(stream);
    return e;
}

}  // namespace ogq

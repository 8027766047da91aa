// Quantize + bit-pack, and unpack + dequantize + sum over K workers.
//
// Both kernels give every CTA a chunk of the flat bucket.  Inside a tensor the unit of work is a group of 128
// (quantizer) or 256 (server) consecutive elements (tensor-relative), which fills a whole number of words; a group belongs
// to the CTA whose chunk holds its first element, so no two ever touch the same word.  Quantizer: lane l
// handles elements 4l..4l+3 (one 128-bit load, one Philox block).  (Runs and level tables of their own for the warps, without
// barriers, were 2 us faster where many small tensors follow one another and 8 to 12 % slower in tensors of 100 M elements.)
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "ogq_common.cuh"
#include "ogq_internal.h"
#include "ogq_quant.cuh"
#include "ogq_unpack.cuh"

namespace ogq {

// CLIP: every value is first clamped to [-tau_arr[t], tau_arr[t]] (gradient clipping).
template <int BITS, bool THRESHOLD, bool CLIP>
__global__ void __launch_bounds__(kThreads, 4)
k_quantize_pack(const float* __restrict__ grad, const int64_t* __restrict__ off, int T, int64_t total,
                int64_t chunk, int s, const float* levels, const float* thresh, const float* tau_arr,
                const __grid_constant__ PhiloxKeys keys, uint32_t stream_id,
                const int64_t* __restrict__ packed_off, uint32_t* __restrict__ packed, const __grid_constant__ QuantSteps steps,
                int early)
{
    __shared__ float sh_lv[kMaxLevels];
    __shared__ float2 sh_tab[kMaxLevels];
    pdl_wait();
    if (early) pdl_launch_dependents();

    const int64_t lo = (int64_t)blockIdx.x * chunk;
    const int64_t hi = (lo + chunk < total) ? lo + chunk : total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kWords = 4 * BITS;  // words of a group

    for_each_piece(off, T, lo, hi, [&](int t, int64_t tb, int64_t te, int64_t pb, int64_t pe) {
        const int64_t n = te - tb;
        const int64_t g_beg = (pb - tb + 127) >> 7, g_end = (pe - tb + 127) >> 7;
        if (g_beg >= g_end) return;
        float b0 = 0.f;
        const float tau = CLIP ? __ldcg(tau_arr + t) : 0.f;
        auto clip = [&](float x) -> float { return CLIP ? copysignf(fminf(fabsf(x), tau), x) : x; };
        bool scales = true;
        if (THRESHOLD) {
            b0 = __ldcg(thresh + t);
        } else {
            __syncthreads();
            bool ok = true;
            if (threadIdx.x < s) {
                const float cur = __ldcg(levels + (int64_t)t * s + threadIdx.x);
                const float nxt = (int)threadIdx.x + 1 < s ? __ldcg(levels + (int64_t)t * s + threadIdx.x + 1) : cur;
                sh_lv[threadIdx.x] = cur;
                sh_tab[threadIdx.x] = quant_table_entry(cur, nxt);
                ok = quant_table_scales(cur, nxt);
            }
            scales = __syncthreads_and(ok);
        }
        const int64_t region = __ldg(packed_off + t + 1) - __ldg(packed_off + t);
        uint32_t* out = packed + __ldg(packed_off + t);
        const bool aligned = (tb & 3) == 0;
        const float* base = grad + tb;

        // Fast path: groups that lie wholly inside the tensor, 128-bit loads (32-bit ones in a tensor that does not
        // start on a 16-byte boundary), kU groups in flight per warp, no bounds checks.  The generic loop below takes
        // what is left: the last, partial group; everything when the tensor's Philox counters do not fit
        // 32 bits or its levels are outside the range of quant_table_scales.
        int64_t g_rest = g_beg;
        if (scales && n <= ((int64_t)1 << 34)) {
            const int64_t g_full = (n >> 7) < g_end ? (n >> 7) : g_end;
            if (g_full > g_beg) {
                g_rest = g_full;
                const int ng = (int)(g_full - g_beg);
                const float* src = base + (g_beg << 7) + 4 * lane;
                uint32_t* dst = out + g_beg * kWords;
                const uint32_t c0_first = (uint32_t)(g_beg << 5) + (uint32_t)lane;  // counters fit 32 bits here
                const uint32_t tabaddr = (uint32_t)__cvta_generic_to_shared(sh_tab);
                float mid = 0.f;
                PhiloxHoist hz = {};
                if constexpr (!THRESHOLD) {
                    mid = sh_tab[(BITS >= 2) ? (1 << (BITS - 2)) : 0].x;
                    hz = philox_hoist(0u, (uint32_t)t, stream_id, keys);
                }
                auto code4 = [&](float4 v, int gl) {
                    if constexpr (CLIP) { v.x = clip(v.x); v.y = clip(v.y); v.z = clip(v.z); v.w = clip(v.w); }
                    uint32_t chunk4;
                    if constexpr (THRESHOLD) {
                        chunk4 = ((v.x >= b0) ? 1u : 0u) | ((v.y >= b0) ? 2u : 0u) | ((v.z >= b0) ? 4u : 0u) | ((v.w >= b0) ? 8u : 0u);
                    } else {
                        const uint4 r = philox4x32_10_tail(c0_first + ((uint32_t)gl << 5), hz, keys);
                        chunk4 = codes_of_entries<BITS>(entry_after_rounding<BITS>(v.x, r.x, tabaddr, mid, steps),
                                                        entry_after_rounding<BITS>(v.y, r.y, tabaddr, mid, steps),
                                                        entry_after_rounding<BITS>(v.z, r.z, tabaddr, mid, steps),
                                                        entry_after_rounding<BITS>(v.w, r.w, tabaddr, mid, steps), tabaddr);
                    }
                    store_chunks<BITS>(dst + (size_t)gl * kWords, chunk4, lane);
                };
                constexpr int kU = 4;  // groups per warp and trip: all loads are issued before the first use
                auto stream = [&](auto vec) {
                    auto load4 = [&](int gl) -> float4 {
                        const float* p = src + (size_t)gl * 128;
                        if constexpr (decltype(vec)::value) return __ldg(reinterpret_cast<const float4*>(p));
                        else return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
                    };
                    const int rest = ng - warp - (kU - 1) * kWarps - 1;
                    const int trips = rest >= 0 ? rest / (kU * kWarps) + 1 : 0;
                    constexpr int kStep = CLIP ? -kU * kWarps : kU * kWarps;
                    int gl = warp + (CLIP ? (trips - 1) * kU * kWarps : 0);
                    for (int k = 0; k < trips; ++k, gl += kStep) {
                        // L2 is asked for the block (kU kWarps groups, 512 bytes each) two trips ahead: the random-rounding
                        // variants compute long enough between their loads for it to pay
                        if (!THRESHOLD && threadIdx.x == 0 && (CLIP ? k + 2 < trips : gl + 3 * kU * kWarps <= ng))
                            prefetch_l2(src - (tb & 3) + (int64_t)(gl + 2 * kStep) * 128, kU * kWarps * 512u);
                        float4 v[kU];
#pragma unroll
                        for (int u = 0; u < kU; ++u) v[u] = load4(gl + u * kWarps);
#pragma unroll
                        for (int u = 0; u < kU; ++u) code4(v[u], gl + u * kWarps);
                    }
                    for (gl = warp + trips * kU * kWarps; gl < ng; gl += kWarps) code4(load4(gl), gl);
                };
                if (aligned) stream(std::true_type());
                else stream(std::false_type());
            }
        }

        for (int64_t g = g_rest + warp; g < g_end; g += kWarps) {
            const int64_t i0 = (g << 7) + 4 * lane;
            float x[4];
            if (aligned && i0 + 3 < n) {
                const float4 v = __ldg(reinterpret_cast<const float4*>(base + i0));
                x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) x[j] = (i0 + j < n) ? __ldg(base + i0 + j) : 0.f;
            }
            if constexpr (CLIP) {
#pragma unroll
                for (int j = 0; j < 4; ++j) x[j] = clip(x[j]);
            }
            uint32_t c[4];
            if (THRESHOLD) {
#pragma unroll
                for (int j = 0; j < 4; ++j) c[j] = (x[j] >= b0) ? 1u : 0u;
            } else {
                const uint64_t q = (uint64_t)i0 >> 2;
                const uint4 r = philox4x32_10((uint32_t)q, (uint32_t)(q >> 32), (uint32_t)t, stream_id, keys);
                const uint32_t rw[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) c[j] = code_as_written<BITS>(x[j], rw[j], [&](int k) { return sh_lv[k]; });
            }
            if (i0 + 3 >= n) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (i0 + j >= n) c[j] = 0u;  // zero padding beyond the tensor
            }
            const uint32_t word = assemble_words<BITS>(c[0] | (c[1] << BITS) | (c[2] << (2 * BITS)) | (c[3] << (3 * BITS)), lane);
            const int64_t widx = g * kWords + packed_word<BITS>(lane);
            if (packs_word<BITS>(lane) && widx < region) out[widx] = word;
        }
    }, CLIP);  // clipped: the threshold's pass went up, the solver's two down and up
}

constexpr size_t kRowsBytes = 16 * 1024;  // level rows of the server step's tensors: 32 tensors of eight workers of nine levels, two of the most
constexpr int kMaxTables = 16;            // and tables of sums

// Server step.  A CTA takes a chunk of the flat bucket, its warps the groups in turn: with a run of its own for every warp
// the workers' streams were read in pieces too short for DRAM (62 instead of 52 us for 25.6 M elements of eight workers,
// nine levels).  The level rows (and tables of sums) of the next `batch` tensors of the chunk are in shared memory at a
// time: their levels lie one after the other in every worker's array, so they come with one wait, and the groups of
// these tensors are gone through without barriers.  (Rows of one tensor at a time, with two barriers and a wait for L2 each,
// and small tensors' levels read from L2 per element: 62 instead of 55 us for nine levels, eight workers and the 161 tensors of the ResNet-50 bucket, 82 instead of 61 for five levels.)
template <int BITS, int REST>
__global__ void __launch_bounds__(kThreads, kStreamCtas)
k_unpack_sum(const uint32_t* const* __restrict__ packed_k, const float* const* __restrict__ levels_k, int K,
             const int64_t* __restrict__ off, const int64_t* __restrict__ packed_off, int T, int64_t total,
             int64_t chunk, int s, int batch, float scale, float* __restrict__ outp)
{
    extern __shared__ __align__(1024) unsigned char sh_mem[];  // tables of sums [kMaxTables][256], then level rows [batch][row_bytes(K)]
    __shared__ const uint32_t* sh_pk[kMaxWorkers];
    __shared__ const float* sh_lv[kMaxWorkers];
    static_assert(kThreads == 256, "a thread per entry of a table");
    constexpr int kWords = 8 * BITS;  // words of a group
    constexpr bool kTable = kTableFloats<BITS> > 0;
    pdl_wait();
    pdl_launch_dependents();

    const int64_t lo = (int64_t)blockIdx.x * chunk;
    const int64_t hi = (lo + chunk < total) ? lo + chunk : total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if ((int)threadIdx.x < (REST < 0 ? 8 : K)) {  // (a table's absent workers read the last one's codes)
        sh_pk[threadIdx.x] = packed_k[min((int)threadIdx.x, K - 1)];
        if ((int)threadIdx.x < K) sh_lv[threadIdx.x] = levels_k[threadIdx.x];
    }
    __syncthreads();
    const uint32_t rb = row_bytes<BITS>(K);
    float* tables = reinterpret_cast<float*>(sh_mem);
    unsigned char* rows = sh_mem + (kTable ? kMaxTables * 1024 : 0);
    int t_first = -1;  // the first tensor whose rows are here
    int turn = 0;      // the warp that takes the next group

    for_each_piece(off, T, lo, hi, [&](int t, int64_t tb, int64_t te, int64_t pb, int64_t pe) {
        const int64_t n = te - tb;
        const int64_t g_beg = (pb - tb + 255) >> 8, g_end = (pe - tb + 255) >> 8;
        if (g_beg >= g_end) return;
        const int64_t pofs = __ldg(packed_off + t);  // (asked for before the rows are waited for)
        if (t_first < 0 || t >= t_first + batch) {
            if (t_first >= 0) __syncthreads();
            t_first = t;
            // row entry `code` of worker k in tensor t + i; codes above s - 1 (never produced by the quantizer) read the top level
            // (of the tensors that begin in this chunk; batch <= 32)
            const int most = batch < T - t ? batch : T - t;
            const int nt = most == 1 ? 1 : __popc(__ballot_sync(0xffffffffu, lane < most && __ldg(off + t + (lane < most ? lane : 0)) < hi));
            if constexpr (kTable) {
                if (nt == 1)  // one tensor: its table from L2 as well, without a barrier in between
                    tables[threadIdx.x] = table_entry<BITS>(threadIdx.x, K, [&](int k, int code) {
                        return __ldcg(sh_lv[k] + (int64_t)t * s + (code < s ? code : s - 1));
                    });
            }
            const int width = 32 - __clz(K - 1) + BITS;  // log2 of the entries per tensor, rounded up
#pragma unroll 4
            for (int i = threadIdx.x; i < nt << width; i += kThreads) {
                const int j = i >> width, q = i & ((1 << width) - 1), k = q >> BITS, code = q & ((1 << BITS) - 1);
                if (k < K)
                    reinterpret_cast<float*>(rows + (size_t)j * rb)[q] = __ldcg(sh_lv[k] + (int64_t)(t + j) * s + (code < s ? code : s - 1));
            }
            __syncthreads();
            if constexpr (kTable) {
                if (nt > 1) {
                    for (int j = 0; j < nt; ++j) {
                        const float* row = reinterpret_cast<const float*>(rows + (size_t)j * rb);
                        tables[j * 256 + threadIdx.x] = table_entry<BITS>(threadIdx.x, K, [&](int k, int code) { return row[(k << BITS) + code]; });
                    }
                    __syncthreads();
                }
            }
        }
        const int all = (int)(g_end - g_beg), first = (warp - turn) & (kWarps - 1);
        turn = (turn + all) & (kWarps - 1);
        if (first >= all) return;
        float* dst = outp + tb;
        const int slot = t - t_first;
        const uint32_t row = (uint32_t)__cvta_generic_to_shared(rows) + (uint32_t)slot * rb,
                       table = (uint32_t)__cvta_generic_to_shared(tables) + (uint32_t)slot * 1024u;
        const int64_t g_full = (n >> 8) < g_end ? (n >> 8) : g_end;
        const int ng = g_full > g_beg ? (int)(g_full - g_beg) : 0;
        const int shift = (int)((reinterpret_cast<uintptr_t>(dst) >> 2) & 3);  // floats above a 16-byte boundary
        const int64_t w0 = pofs + g_beg * kWords;
        float* dst8 = dst + (g_beg << 8) + 8 * lane;
        auto write = [&](int gl, float (&a)[8]) {
#pragma unroll
            for (int j = 0; j < 8; ++j) a[j] = __fmul_rn(a[j], scale);
            store8<(BITS > 1)>(dst8 + (size_t)gl * 256, shift, lane, a);
        };
        constexpr int G = 2;       // groups per warp and trip
        constexpr int kAhead = 8;  // trips between two prefetch requests
        constexpr int kTrip = G * kWarps;
        int gl = first;
        if constexpr (REST < 0) {
            // 1-bit codes of a few workers: a warp takes four groups in a row, whose codes are one word per lane and worker, and gets a
            // group's bytes from the lanes that have them.
            constexpr int N = REST == kTableOnly ? 8 : 4;  // (codes of workers that do not exist mean nothing to the table)
            const int quads = ng >> 2;
            uint32_t next[N];
            auto load = [&](int q) {
#pragma unroll
                for (int u = 0; u < N; ++u) next[u] = __ldcg(sh_pk[u] + w0 + (int64_t)q * 32 + lane);
            };
            int q = first;
            if (q < quads) load(q);
            for (; q < quads; q += kWarps) {
                uint32_t w[N];
#pragma unroll
                for (int u = 0; u < N; ++u) w[u] = next[u];
                if (q + kWarps < quads) load(q + kWarps);
#pragma unroll 1
                for (int g = 0; g < 4; ++g) {
                    uint32_t c[kTableWorkers<BITS>], x[2];
#pragma unroll
                    for (int u = 0; u < kTableWorkers<BITS>; ++u)
                        c[u] = u < N ? __byte_perm(__shfl_sync(0xffffffffu, w[u < N ? u : 0], 8 * g + (lane >> 2)), 0u, 0x4440 + (lane & 3)) : 0u;
                    table_indices<BITS>(c, x);
                    float a[8];
                    read_table(x, table, a);
                    write(4 * q + g, a);
                }
            }
            gl = 4 * quads + first;
        }
        for (int trip = 0; REST >= 0 && gl + kWarps < ng; gl += kTrip, ++trip) {
            // every kAhead trips K threads ask L2 for the workers' words of the kAhead trips after the next
            // kAhead (no gain at one bit per code)
            if (BITS >= 2 && (trip & (kAhead - 1)) == 0 && (int)threadIdx.x < K && (trip + 2 * kAhead) * kTrip <= ng)
                prefetch_l2(sh_pk[threadIdx.x] + w0 + (int64_t)(trip + kAhead) * kTrip * kWords, kAhead * kTrip * kWords * 4u);
            float a[G][8];
            sum_workers<BITS, G, true, REST>(K, lane, table, row,
                                 [&](int k, int g) { return sh_pk[k] + w0 + (int64_t)(gl + g * kWarps) * kWords; }, a);
#pragma unroll
            for (int g = 0; g < G; ++g) write(gl + g * kWarps, a[g]);
        }
        if (gl < ng) {
            float a[1][8];
            sum_workers<BITS, 1, true, REST>(K, lane, table, row, [&](int k, int) { return sh_pk[k] + w0 + (int64_t)gl * kWords; }, a);
            write(gl, a[0]);
        }

        // the tensor's last, partial group
        if (all > ng && ((ng - first) & (kWarps - 1)) == 0) {
            const int64_t i0 = (g_full << 8) + 8 * lane;
            if (i0 < n) {
                const int64_t region = __ldg(packed_off + t + 1) - pofs, wi = (i0 * BITS) >> 5;
                const int sh = (int)(i0 * BITS) & 31;
                const bool two = sh + 8 * BITS > 32 && wi + 1 < region;
                const float* mine = reinterpret_cast<const float*>(rows + (size_t)slot * rb);
                float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
                for (int k = 0; k < K; ++k) {
                    const uint32_t* p = sh_pk[k] + pofs + wi;
                    const uint32_t a = __ldcg(p), b = two ? __ldcg(p + 1) : 0u;
                    const uint64_t codes = ((uint64_t)b << 32 | a) >> sh;
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        acc[j] = __fadd_rn(acc[j], mine[(k << BITS) + ((int)(codes >> (j * BITS)) & ((1 << BITS) - 1))]);
                }
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (i0 + j < n) dst[i0 + j] = __fmul_rn(acc[j], scale);
            }
        }
    });
}

// Server step of one worker.  Nothing is summed, so a warp keeps a tensor's levels in a register of its lanes and looks a code up
// with a shuffle: no shared memory and no barrier, and the levels are asked for at the same time as the codes.  Small buckets
// wait for L2 once instead of twice, large ones are bounded by DRAM.  Kernel above with one worker, and this one: 50,000
// elements of one tensor 3.0 and 2.4 us (two levels), 300,000 in 60 tensors 7.3 and 5.0, the ResNet-50 bucket 32.7 and 23.8
// (nine levels: 30.2 and 23.3), 70 M elements of nine levels 61.5 and 57.1.
template <int BITS>
__global__ void __launch_bounds__(kThreads, kStreamCtas)
k_unpack_one(const uint32_t* const* __restrict__ packed_k, const float* const* __restrict__ levels_k, const int64_t* __restrict__ off,
             const int64_t* __restrict__ packed_off, int T, int64_t total, int64_t chunk, int s, float scale, float* __restrict__ outp)
{
    constexpr int kWords = 8 * BITS;  // words of a group
    pdl_wait();
    pdl_launch_dependents();
    const int64_t lo = (int64_t)blockIdx.x * chunk;
    const int64_t hi = (lo + chunk < total) ? lo + chunk : total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t* pk = packed_k[0];
    const float* lv = levels_k[0];
    int turn = 0;  // the warp that takes the next group
    for_each_piece(off, T, lo, hi, [&](int t, int64_t tb, int64_t te, int64_t pb, int64_t pe) {
        const int64_t n = te - tb;
        const int64_t g_beg = (pb - tb + 255) >> 8, g_end = (pe - tb + 255) >> 8;
        if (g_beg >= g_end) return;
        const int all = (int)(g_end - g_beg), first = (warp - turn) & (kWarps - 1);
        turn = (turn + all) & (kWarps - 1);
        if (first >= all) return;
        // (codes above s - 1, never produced by the quantizer, read the top level; a sum of one term has no negative zero)
        const float level = __fadd_rn(0.f, __ldcg(lv + (int64_t)t * s + (lane < s ? lane : s - 1)));
        const int64_t pofs = __ldg(packed_off + t);
        float* dst = outp + tb;
        const int64_t g_full = (n >> 8) < g_end ? (n >> 8) : g_end;
        const int ng = g_full > g_beg ? (int)(g_full - g_beg) : 0;
        const int shift = (int)((reinterpret_cast<uintptr_t>(dst) >> 2) & 3);  // floats above a 16-byte boundary
        const uint32_t* words = pk + pofs + g_beg * kWords;
        float* dst8 = dst + (g_beg << 8) + 8 * lane;
        auto look_up = [&](const EightCodes<BITS>& c, float (&a)[8]) {
            const uint64_t codes = (uint64_t)c.hi << 32 | c.lo;
#pragma unroll
            for (int j = 0; j < 8; ++j) a[j] = __fmul_rn(__shfl_sync(0xffffffffu, level, (int)(codes >> (j * BITS)) & ((1 << BITS) - 1)), scale);
        };
        // groups whose codes are loaded before any is used (70 M elements: two, four, eight groups 61.4, 57.4 and 59.3 us at one bit,
        // 57.1, 62.6 and 61.9 at four)
        constexpr int G = BITS == 1 ? 4 : 2;
        for (int gl = first; gl < ng; gl += G * kWarps) {
            EightCodes<BITS> c[G];
#pragma unroll
            for (int g = 0; g < G; ++g)
                if (gl + g * kWarps < ng) c[g] = load_codes<BITS>(words + (int64_t)(gl + g * kWarps) * kWords, lane);
#pragma unroll
            for (int g = 0; g < G; ++g) {
                if (gl + g * kWarps >= ng) break;
                float a[8];
                look_up(c[g], a);
                store8<(BITS > 1)>(dst8 + (size_t)(gl + g * kWarps) * 256, shift, lane, a);
            }
        }
        // the tensor's last, partial group
        if (all > ng && ((ng - first) & (kWarps - 1)) == 0) {
            const int64_t i0 = (g_full << 8) + 8 * lane, region = __ldg(packed_off + t + 1) - pofs, wi = (i0 * BITS) >> 5;
            const int sh = (int)(i0 * BITS) & 31;
            const uint32_t a = i0 < n ? __ldcg(pk + pofs + wi) : 0u;
            const uint32_t b = i0 < n && sh + 8 * BITS > 32 && wi + 1 < region ? __ldcg(pk + pofs + wi + 1) : 0u;
            const uint64_t codes = ((uint64_t)b << 32 | a) >> sh;
            EightCodes<BITS> c;
            c.lo = (uint32_t)codes;
            c.hi = (uint32_t)(codes >> 32);
            float x[8];
            look_up(c, x);
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (i0 + j < n) dst[i0 + j] = x[j];
        }
    });
}

cudaError_t launch_quantize_pack(const float* d_grad, const int64_t* d_off, int T, int64_t total,
                                 int scheme, int s, const float* d_levels, const float* d_thresh,
                                 const float* d_tau, uint64_t seed, uint32_t stream_id,
                                 const int64_t* d_packed_off, uint32_t* d_packed, int sm_count,
                                 cudaStream_t stream)
{
    // One wave for the threshold quantizer, whose CTAs then begin where a pass over the same chunks left the data in L2 (97 -> 91 us
    // for 143.7 M elements); three waves for the random ones, which are bound by instruction issue and gain more from
    // an even finish (203, 195, 191, 193, 196 us with one, two, three, four, eight).
    const FlatGrid g = make_flat_grid(total, sm_count * kStreamCtas * (scheme == OGQ_BINGRAD_B ? 1 : 3), 8192);
    const PhiloxKeys keys = philox_round_keys((uint32_t)seed, (uint32_t)(seed >> 32));
    const int bits = ogq_bits_for_levels(s);
    // What follows a threshold quantizer of a full wave is launched when its CTAs end: the next worker's first pass would otherwise
    // share the SMs out unevenly (see kBbAloneN; ResNet-50 bucket in one bit, one worker after the other: 68.1 and 67.1 us each).
    const int early = scheme != OGQ_BINGRAD_B || g.ctas <= sm_count * (kStreamCtas - 1) ? 1 : 0;
    cudaError_t e = cudaErrorInvalidValue;
#define OGQ_LAUNCH_QC(B, TH, CL)                                                                        \
    e = launch_pdl(k_quantize_pack<B, TH, CL>, g.ctas, kThreads, 0, stream, d_grad, d_off, T, total, g.chunk, s, \
                   d_levels, d_thresh, d_tau, keys, stream_id, d_packed_off, d_packed, quant_steps(), early)
#define OGQ_LAUNCH_Q(B, TH)                    \
    do {                                       \
        if (d_tau) OGQ_LAUNCH_QC(B, TH, true); \
        else OGQ_LAUNCH_QC(B, TH, false);      \
    } while (0)
    launch_begin(scheme == OGQ_BINGRAD_B ? "k_quantize_pack_threshold" : "k_quantize_pack_random", stream);
    if (scheme == OGQ_BINGRAD_B) {
        OGQ_LAUNCH_Q(1, true);
    } else {
        switch (bits) {
            case 1: OGQ_LAUNCH_Q(1, false); break;
            case 2: OGQ_LAUNCH_Q(2, false); break;
            case 3: OGQ_LAUNCH_Q(3, false); break;
            case 4: OGQ_LAUNCH_Q(4, false); break;
            case 5: OGQ_LAUNCH_Q(5, false); break;
            default: return cudaErrorInvalidValue;
        }
    }
#undef OGQ_LAUNCH_Q
#undef OGQ_LAUNCH_QC
    launch_end(stream);
    return e;
}

cudaError_t launch_unpack_sum(const uint32_t* const* d_packed_k, const float* const* d_levels_k, int K,
                              const int64_t* d_off, const int64_t* d_packed_off, int T, int64_t total,
                              int s, float scale, float* d_out, int sm_count, cudaStream_t stream)
{
    const FlatGrid g = make_flat_grid(total, sm_count * kStreamCtas, 4096);
    const int bits = ogq_bits_for_levels(s);
    // 1-bit codes, four groups of a tensor at a time, where a CTA has many of one (VGG-19 bucket, eight workers: 180 -> 131 us; 5 M elements
    // 10.1 -> 8.8): many small tensors want their groups shared out more evenly (3 M in 50, five workers: 9.4 against 10.9).
    const bool quads = total / (g.ctas + T) >= 8192;
    cudaError_t e = cudaErrorInvalidValue;
#define OGQ_LAUNCH_U(B)                                                                               \
    if (K == 1) { /* faster at every size and width measured, see the kernel */                       \
        e = launch_pdl(k_unpack_one<B>, g.ctas, kThreads, 0, stream, d_packed_k, d_levels_k, d_off,   \
                       d_packed_off, T, total, g.chunk, s, scale, d_out);                             \
    } else {                                                                                          \
        const size_t each = row_bytes<B>(K), tables = kTableFloats<B> > 0 ? kMaxTables * 1024 : 0;       \
        const int batch = (int)std::min<size_t>(std::max<size_t>(kRowsBytes / each, 1), (size_t)std::min(T, tables ? kMaxTables : 32)); \
        e = with_rest<B, true>(rest_of<B, true>(K, quads), [&](auto rest) {                                         \
            return launch_pdl(k_unpack_sum<B, decltype(rest)::value>, g.ctas, kThreads, tables + each * batch, stream, d_packed_k, \
                              d_levels_k, K, d_off, d_packed_off, T, total, g.chunk, s, batch, scale, d_out); \
        });                                                                                           \
    }
    launch_begin("k_unpack_sum", stream);
    switch (bits) {
        case 1: OGQ_LAUNCH_U(1); break;
        case 2: OGQ_LAUNCH_U(2); break;
        case 3: OGQ_LAUNCH_U(3); break;
        case 4: OGQ_LAUNCH_U(4); break;
        case 5: OGQ_LAUNCH_U(5); break;
        default: return cudaErrorInvalidValue;
    }
#undef OGQ_LAUNCH_U
    launch_end(stream);
    return e;
}

}  // namespace ogq

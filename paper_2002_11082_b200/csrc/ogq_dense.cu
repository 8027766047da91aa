// Entropy-dense wire format: M consecutive codes are the base-s digits of one 32-bit word (least
// significant first), M the largest count with s^M <= 2^32: 20 codes per word for s = 3, 13 for
// s = 5, 10 for s = 9, 7 for s = 17, i.e. 1.6 / 2.46 / 3.2 / 4.57 bits per element instead of
// 2 / 3 / 4 / 5.  The paper's compression ratios (x20.2, x13.8, x10.1) assume log2(s) bits per code;
// this is the closest whole-word format.  Quantization itself (segment search, Philox draw, rounding
// decision) is the one of the bit-packed path: only the packing differs.
//
// Quantizer: a group of U = lcm(4, M) consecutive elements of a tensor is a whole number of 128-bit loads and
// Philox blocks (U / 4) and of output words (U / M).  A warp takes a tile of 32 groups: it loads and codes them 128
// elements at a time, as the bit-packed path does, leaves the codes as bytes in shared memory, and then every lane makes the
// words of one group.  Server: a lane takes one word of every worker, a warp 32 consecutive words, and the
// sums go through shared memory to whole-line stores.  Groups (four words) belong to the CTA whose chunk holds their
// first element.
#include <math.h>

#include <type_traits>

#include "ogq_common.cuh"
#include "ogq_internal.h"
#include "ogq_quant.cuh"
#include "ogq_unpack.cuh"

namespace ogq {

template <int S> struct Dense;
template <> struct Dense<3>  { static constexpr int M = 20, U = 20, BITS = 2; };
template <> struct Dense<5>  { static constexpr int M = 13, U = 52, BITS = 3; };
template <> struct Dense<9>  { static constexpr int M = 10, U = 20, BITS = 4; };
template <> struct Dense<17> { static constexpr int M = 7,  U = 28, BITS = 5; };

__host__ __device__ constexpr uint32_t dense_pow(int s, int q)
{
    uint32_t p = 1;
    for (int i = 0; i < q; ++i) p *= (uint32_t)s;
    return p;
}

int dense_digits(int s)
{
    switch (s) {
        case 3: return 20;
        case 5: return 13;
        case 9: return 10;
        case 17: return 7;
        default: return 0;
    }
}

// The words of one group from its codes, four per 32-bit word x[q] as bytes: sums of four (byte) or two (16-bit weights) products
// at a time.
template <int S>
__device__ __forceinline__ void dense_words(const uint32_t (&x)[Dense<S>::U / 4], uint32_t (&word)[Dense<S>::U / Dense<S>::M])
{
    constexpr int M = Dense<S>::M, Q = Dense<S>::U / 4, W = Dense<S>::U / M;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        word[w] = 0u;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int e = 4 * q - w * M;  // digit of the first of the four codes; those outside [0, M) are another word's
            if (e <= -4 || e >= M) continue;
            const int first = e < 0 ? 0 : e;
            uint32_t c[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) c[j] = e + j >= first && e + j < M ? dense_pow(S, e + j - first) : 0u;
            uint32_t four;
            if constexpr (S <= 5) four = __dp4a(x[q], c[0] | c[1] << 8 | c[2] << 16 | c[3] << 24, 0u);
            else four = __dp2a_lo(c[0] | c[1] << 16, x[q], __dp2a_hi(c[2] | c[3] << 16, x[q], 0u));
            word[w] += four * dense_pow(S, first);
        }
    }
}

// What bounds it: instruction issue, as the bit-packed quantizer.  One lane per group, reading its U elements itself,
// spread each load over 32 lines and took 86 us for 25.6 M elements at s = 5.
template <int S>
__global__ void __launch_bounds__(kThreads, 4)
k_quantize_pack_dense(const float* __restrict__ grad, const int64_t* __restrict__ off, int T, int64_t total, int64_t chunk,
                      const float* levels, const __grid_constant__ PhiloxKeys keys,
                      uint32_t stream_id, const int64_t* __restrict__ packed_off, uint32_t* __restrict__ packed,
                      const __grid_constant__ QuantSteps steps)
{
    constexpr int M = Dense<S>::M, U = Dense<S>::U, BITS = Dense<S>::BITS, W = U / M, Q = U / 4;
    __shared__ float2 sh_tables[kWarps][kMaxLevels];
    __shared__ uint32_t sh_codes[kWarps][32 * Q];
    pdl_wait();
    pdl_launch_dependents();

    const int64_t lo = (int64_t)blockIdx.x * chunk;
    const int64_t hi = (lo + chunk < total) ? lo + chunk : total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float2* sh_tab = sh_tables[warp];
    uint32_t* codes = sh_codes[warp];
    int turn = 0;  // the warp that takes the first tile of the next piece

    for_each_piece(off, T, lo, hi, [&](int t, int64_t tb, int64_t te, int64_t pb, int64_t pe) {
        const int64_t n = te - tb;
        const int64_t g_beg = (pb - tb + U - 1) / U, g_end = (pe - tb + U - 1) / U;
        if (g_beg >= g_end) return;
        const int64_t g_full = (n / U) < g_end ? (n / U) : g_end;  // groups wholly inside the tensor
        const int ng = (int)(g_full - g_beg);
        // the warps take tiles in turn, the words of a partial group or of the padding count as one more; no barriers
        const bool last = g_end == (n + U - 1) / U;
        const int tiles = (ng + 31) / 32, all = tiles + (last ? 1 : 0), first = (warp - turn) & (kWarps - 1);
        turn = (turn + all) & (kWarps - 1);
        if (first >= all) return;
        bool ok = true;
        __syncwarp();
        if (lane < S) {
            const float cur = __ldcg(levels + (int64_t)t * S + lane);
            const float nxt = lane + 1 < S ? __ldcg(levels + (int64_t)t * S + lane + 1) : cur;
            sh_tab[lane] = quant_table_entry(cur, nxt);
            ok = quant_table_scales(cur, nxt);
        }
        __syncwarp();
        const bool scales = __all_sync(0xffffffffu, ok);
        const int64_t region = __ldg(packed_off + t + 1) - __ldg(packed_off + t);
        uint32_t* out = packed + __ldg(packed_off + t);
        const float* base = grad + tb;

        int i_rest = first;
        if (scales && n <= ((int64_t)1 << 34)) {
            if (first < tiles) {
                i_rest = first + (tiles - first + kWarps - 1) / kWarps * kWarps;  // this warp's first tile that is not done
                const uint32_t tabaddr = (uint32_t)__cvta_generic_to_shared(sh_tab);
                const float mid = sh_tab[1 << (BITS - 2)].x;
                const PhiloxHoist hz = philox_hoist(0u, (uint32_t)t, stream_id, keys);
                const float* src = base + g_beg * U + 4 * lane;
                const uint32_t c0_first = (uint32_t)(g_beg * Q) + (uint32_t)lane;
                auto tile = [&](int g0, auto vec, auto all) {
                    constexpr bool whole = decltype(all)::value;  // all 32 groups are there
                    constexpr int B = 4;  // loads in flight
                    const int quads = whole ? 32 * Q : (ng - g0) * Q;
                    const float* p = src + (size_t)g0 * U;
#pragma unroll
                    for (int q0 = 0; q0 < Q; q0 += B) {
                        float4 v[B];
#pragma unroll
                        for (int u = 0; u < B; ++u) {
                            if (q0 + u < Q && (whole || (q0 + u) * 32 + lane < quads)) {
                                const float* a = p + (q0 + u) * 128;
                                if constexpr (decltype(vec)::value) v[u] = __ldg(reinterpret_cast<const float4*>(a));
                                else v[u] = make_float4(__ldg(a), __ldg(a + 1), __ldg(a + 2), __ldg(a + 3));
                            } else {
                                v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                            }
                        }
#pragma unroll
                        for (int u = 0; u < B; ++u) {
                            if (q0 + u >= Q) continue;
                            const uint4 r = philox4x32_10_tail(c0_first + (uint32_t)(g0 * Q + (q0 + u) * 32), hz, keys);
                            codes[(q0 + u) * 32 + lane] =
                                codes_of_entries<8>(entry_after_rounding<BITS>(v[u].x, r.x, tabaddr, mid, steps),
                                                    entry_after_rounding<BITS>(v[u].y, r.y, tabaddr, mid, steps),
                                                    entry_after_rounding<BITS>(v[u].z, r.z, tabaddr, mid, steps),
                                                    entry_after_rounding<BITS>(v[u].w, r.w, tabaddr, mid, steps), tabaddr);
                        }
                    }
                    __syncwarp();
                    uint32_t x[Q], word[W];
#pragma unroll
                    for (int q = 0; q < Q; ++q) x[q] = codes[lane * Q + q];
                    __syncwarp();
                    dense_words<S>(x, word);
                    if (whole || g0 + lane < ng) {
                        uint32_t* dst = out + (g_beg + g0 + lane) * W;
                        if constexpr (W == 1) dst[0] = word[0];
                        else if constexpr (W == 2) *reinterpret_cast<uint2*>(dst) = make_uint2(word[0], word[1]);
                        else *reinterpret_cast<uint4*>(dst) = make_uint4(word[0], word[1], word[2], word[3]);
                    }
                };
                auto stream = [&](auto vec) {
                    int g0 = first * 32;
                    for (; g0 + 32 <= ng; g0 += kWarps * 32) tile(g0, vec, std::true_type());
                    if (g0 < ng) tile(g0, vec, std::false_type());
                };
                if ((tb & 3) == 0) stream(std::true_type());
                else stream(std::false_type());
            }
        }

        // generic path: one lane per output word, element by element (the last, partial group; everything when
        // the tensor's Philox counters do not fit 32 bits or its levels are outside the range of quant_table_scales)
        // (the warp that takes the last tile also writes the zero padding of the region)
        for (; i_rest < all; i_rest += kWarps) {
          const int64_t w_beg = (i_rest < tiles ? g_beg + (int64_t)i_rest * 32 : g_full) * W;
          const int64_t w_end = i_rest >= tiles ? region : (i_rest * 32 + 32 < ng ? w_beg + 32 * W : g_full * W);
          for (int64_t wi = w_beg + lane; wi < w_end; wi += 32) {
            uint32_t word = 0u, p = 1u;
            for (int d = 0; d < M; ++d) {
                const int64_t i = wi * M + d;
                if (i < n) {
                    const float x = __ldg(base + i);
                    const uint64_t blk = (uint64_t)i >> 2;
                    const uint4 r = philox4x32_10((uint32_t)blk, (uint32_t)(blk >> 32), (uint32_t)t, stream_id, keys);
                    const uint32_t rnd = (i & 3) == 0 ? r.x : ((i & 3) == 1 ? r.y : ((i & 3) == 2 ? r.z : r.w));
                    word += code_as_written<BITS>(x, rnd, [&](int k) { return sh_tab[k].x; }) * p;
                }
                p *= (uint32_t)S;
            }
            out[wi] = word;
          }
        }
    });
}

// A word w as the fraction w / S^M, in units of 2^-32: multiplied by S, its integer part is the word's highest digit and
// the rest the fraction of the remaining word, so every further digit is one wide multiplication.  Any
// f in [w R, (w + 1) R), R = 2^32 / S^M, gives the right digits: no multiple of a power of S lies between the two ends.  w R
// is taken as w floor(R) + w C / 2^32 + 1, rounded down, C / 2^32 the fraction of R: for S = 5 and 17, C rounded up is
// good enough (R > 2); for 3^20 = 9^10, R = 1.23, and C needs its first binary place behind the point, too.
template <int S>
__device__ __forceinline__ uint32_t dense_fraction(uint32_t w)
{
    if constexpr (S == 5) return __umulhi(w, 2226670858u) + 3u * w + 1u;
    else if constexpr (S == 17) return __umulhi(w, 2005251564u) + 10u * w + 1u;
    else return (uint32_t)(((uint64_t)w * 995507236u + ((w >> 1) + 1u)) >> 32) + w + 1u;
}

// A worker's row of levels for D digits at a time: D tables of S^D entries, table a that of the a-th of the D digits (the highest
// first) in the number that the D digits make.  Entries of one table lie in different banks, S^D <= 32.
template <int S, int D>
struct DenseRow {
    static constexpr int kEntries = (int)dense_pow(S, D), kFloats = D * kEntries, kPlain = (D - 1) * kEntries;  // kPlain: the levels themselves
    static_assert(D == 1 || kEntries <= 32, "no bank conflicts");
};

// acc[e] += the level of digit e of w.  row: shared address of the worker's row.
template <int S, int D>
__device__ __forceinline__ void add_digits(uint32_t w, uint32_t row, float (&acc)[Dense<S>::M])
{
    constexpr int M = Dense<S>::M, E = DenseRow<S, D>::kEntries;
    uint32_t f = dense_fraction<S>(w);
    float v[M];
#pragma unroll
    for (int e = M - 1; e >= 0; e -= D) {
        constexpr int kLeft = M % D == 0 ? D : M % D;  // digits of the last step
        const int r = e + 1 < D ? kLeft : D;
        uint32_t at;
        asm("{ .reg .b64 p; .reg .b32 d; mul.wide.u32 p, %1, %2; mov.b64 {%1, d}, p; mad.lo.u32 %0, d, 4, %3; }"
            : "=r"(at), "+r"(f) : "r"(dense_pow(S, r)), "r"(row));
#pragma unroll
        for (int i = 0; i < D; ++i)
            if (i < r) asm("ld.shared.f32 %0, [%1];" : "=f"(v[e - i >= 0 ? e - i : 0]) : "r"(at + (uint32_t)((D - r + i) * E * 4)));
    }
#pragma unroll
    for (int e = 0; e + 1 < M; e += 2) add2(acc[e], acc[e + 1], v[e], v[e + 1]);
    if constexpr (M & 1) acc[M - 1] = __fadd_rn(acc[M - 1], v[M - 1]);
}

// The rows of K workers for tensor t, by `warps` warps of which this is number w; sync: their barrier.
template <int S, int D, class Sync>
__device__ __forceinline__ void dense_rows(float* rows, const float* const* lv, int K, int64_t t, int w, int warps, Sync sync)
{
    using Row = DenseRow<S, D>;
    const int lane = threadIdx.x & 31;
    if constexpr (D == 2) {
        // A warp has a worker or a few to itself: both tables straight from the levels, one wait and one barrier.  (With three
        // tables, and with one warp for all workers, it is no faster: 1 % and 3 % more for eight workers.)
        if (warps > 1) {
            if (lane < Row::kEntries) {
                for (int k = w; k < K; k += warps) {
                    const float* l = lv[k] + t * S;
                    float* row = rows + k * Row::kFloats;
                    row[lane] = __ldcg(l + lane / S);
                    row[Row::kEntries + lane] = __ldcg(l + lane % S);
                }
            }
            sync();
            return;
        }
    }
    for (int i = w * 32 + lane; i < K * S; i += warps * 32) rows[i / S * Row::kFloats + Row::kPlain + i % S] = __ldcg(lv[i / S] + t * S + i % S);
    sync();
    if constexpr (D > 1) {
        // entry `lane` of every table, from the levels themselves, which are the first entries of the last
        if (lane < Row::kEntries) {
#pragma unroll 4
            for (int k = w; k < K; k += warps) {
                float* row = rows + k * Row::kFloats;
#pragma unroll
                for (int a = 0; a < D; ++a) {
                    const float x = row[Row::kPlain + (uint32_t)lane / dense_pow(S, D - 1 - a) % S];
                    if (a + 1 < D || lane >= S) row[a * Row::kEntries + lane] = x;
                }
            }
        }
        sync();
    }
}

// Workers whose words the server step asks for before it uses any.
template <int S> constexpr int kDenseBatch = Dense<S>::M == 20 ? 2 : 4;

// What bounds it: shared-memory reads, one per element and worker, with the instructions for the digits close behind: a wide product
// holds the multiply pipe for four cycles.  So three digits at a time (S = 3) or two (S = 5) come from one product and one address,
// each with a read of a table of its own, as long as four CTAs' tables fit an SM (25.6 M elements of eight workers at S = 5, whole
// step: 204 -> 198 us; 20 M at S = 3: 49 -> 41).  (One lane per group with divisions by S and stores of its own, each spread over 32 lines: 119 us for 25.6 M
// elements of 8 workers at s = 5.)  Two digits at a time through one table of pairs were no faster: a 64-bit
// read costs as much as two.
// REST: number of workers in the last, partial batch.  They are loaded together as those of a full one, and as a template argument
// it leaves no condition between them (25 M elements in 161 tensors, two and three workers, one after the other before: S = 5 37 -> 31
// and 47 -> 35 us, S = 9 46 -> 35 and 58 -> 42; seven workers of nine levels 87 -> 73).  With a loop over the number instead, the full
// batches of S = 9 get slower (eight workers 76 -> 83 us).
template <int S, int D, int REST>
__global__ void __launch_bounds__(kThreads, 4)
k_unpack_sum_dense(const uint32_t* const* __restrict__ packed_k, const float* const* __restrict__ levels_k, int K,
                   const int64_t* __restrict__ off, const int64_t* __restrict__ packed_off, int T, int64_t total,
                   int64_t chunk, float scale, float* __restrict__ outp)
{
    constexpr int M = Dense<S>::M, U = 4 * M;  // U: elements of a group here (whole 16-byte lines whatever M)
    constexpr int kTile = 32 * M;              // elements of a tile
    constexpr int kEdgeTiles = 4;              // tensors of no more tiles in this chunk go to one warp each
    constexpr int kRow = DenseRow<S, D>::kFloats;
    extern __shared__ __align__(16) float sh_sums[];  // [kWarps][kTile] sums, then [kWarps + 2][K][kRow] level rows
    __shared__ const uint32_t* sh_pk[kMaxWorkers];
    __shared__ const float* sh_lv[kMaxWorkers];
    pdl_wait();
    pdl_launch_dependents();

    const int64_t lo = (int64_t)blockIdx.x * chunk;
    const int64_t hi = (lo + chunk < total) ? lo + chunk : total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if ((int)threadIdx.x < K) {
        sh_pk[threadIdx.x] = packed_k[threadIdx.x];
        sh_lv[threadIdx.x] = levels_k[threadIdx.x];
    }
    __syncthreads();
    float* sum = sh_sums + warp * kTile;
    float* all_rows = sh_sums + kWarps * kTile;
    int turn = 0;  // the warp that takes the next small tensor
    int set = 0;   // of the two sets of rows of larger ones: a warp that is done with one may fill the other

    for_each_piece(off, T, lo, hi, [&](int t, int64_t tb, int64_t te, int64_t pb, int64_t pe) {
        const int64_t n = te - tb;
        const int64_t g_beg = (pb - tb + U - 1) / U, g_end = (pe - tb + U - 1) / U;
        if (g_beg >= g_end) return;
        const int64_t pofs = __ldg(packed_off + t);
        const int64_t w_beg = g_beg * 4;
        const int64_t w_all = (n + M - 1) / M, w_end = g_end * 4 < w_all ? g_end * 4 : w_all;
        const int tiles = (int)((w_end - w_beg + 31) / 32);
        const bool vec = (reinterpret_cast<uintptr_t>(outp + tb) & 15) == 0;

        const bool small = tiles <= kEdgeTiles;
        float* rows = all_rows + (small ? warp : kWarps + set) * K * kRow;
        if (small) {
            turn = (turn + 1) & (kWarps - 1);
            if (turn != warp) return;
            __syncwarp();
            dense_rows<S, D>(rows, sh_lv, K, t, 0, 1, [] { __syncwarp(); });
        } else {
            set ^= 1;
            dense_rows<S, D>(rows, sh_lv, K, t, warp, kWarps, [] { __syncthreads(); });
        }
        const uint32_t rows_addr = (uint32_t)__cvta_generic_to_shared(rows);
        const int first = small ? 0 : warp, step = small ? 1 : kWarps;
        for (int i = first; i < tiles; i += step) {  // a word of every worker per lane
            const int64_t w0 = w_beg + (int64_t)i * 32;
            const bool have = w0 + lane < w_end;
            const int64_t at = pofs + w0 + lane;
            // every kAhead trips the first K threads ask L2 for the workers' words of the kAhead trips after the next kAhead
            constexpr int kAhead = 8;
            if (((i / kWarps) & (kAhead - 1)) == 0 && (int)threadIdx.x < K && i + 2 * kAhead * kWarps <= tiles - 1)
                prefetch_l2(sh_pk[threadIdx.x] + pofs + w_beg + (int64_t)(i / kWarps + kAhead) * kWarps * 32, kAhead * kWarps * 128u);
            float acc[M];
#pragma unroll
            for (int e = 0; e < M; ++e) acc[e] = 0.f;
            constexpr int B = kDenseBatch<S>;
            auto batch = [&](auto count, int k) {
                constexpr int N = decltype(count)::value;
                uint32_t w[N];
#pragma unroll
                for (int u = 0; u < N; ++u) w[u] = have ? __ldcg(sh_pk[k + u] + at) : 0u;
#pragma unroll
                for (int u = 0; u < N; ++u) add_digits<S, D>(w[u], rows_addr + (k + u) * (kRow * 4), acc);
            };
            for (int k = 0; k + B <= K; k += B) batch(std::integral_constant<int, B>{}, k);
            if constexpr (REST > 0) batch(std::integral_constant<int, REST>{}, K - REST);
#pragma unroll
            for (int e = 0; e < M; ++e) acc[e] = __fmul_rn(acc[e], scale);
            float* mine = sum + lane * M;  // no bank conflicts at any of these strides and widths
            if constexpr (M % 4 == 0) {
#pragma unroll
                for (int e = 0; e < M; e += 4) *reinterpret_cast<float4*>(mine + e) = make_float4(acc[e], acc[e + 1], acc[e + 2], acc[e + 3]);
            } else if constexpr (M % 2 == 0) {
#pragma unroll
                for (int e = 0; e < M; e += 2) *reinterpret_cast<float2*>(mine + e) = make_float2(acc[e], acc[e + 1]);
            } else {
#pragma unroll
                for (int e = 0; e < M; ++e) mine[e] = acc[e];
            }
            __syncwarp();
            const int64_t e0 = w0 * M, left = (w_end * M < n ? w_end * M : n) - e0;
            float* dst = outp + tb + e0;
            if (vec && left >= kTile) {
#pragma unroll
                for (int e = 0; e < kTile; e += 128)
                    if (e + 128 <= kTile || e + 4 * lane < kTile)
                        *reinterpret_cast<float4*>(dst + e + 4 * lane) = *reinterpret_cast<const float4*>(sum + e + 4 * lane);
            } else {
#pragma unroll 4
                for (int e = lane; e < kTile; e += 32)
                    if (e < left) dst[e] = sum[e];
            }
            __syncwarp();
        }
    });
}

cudaError_t launch_quantize_pack_dense(const float* d_grad, const int64_t* d_off, int T, int64_t total, int s,
                                       const float* d_levels, uint64_t seed, uint32_t stream_id,
                                       const int64_t* d_packed_off, uint32_t* d_packed, int sm_count,
                                       cudaStream_t stream)
{
    const FlatGrid g = make_flat_grid(total, sm_count * kStreamCtas, 4096);
    const PhiloxKeys keys = philox_round_keys((uint32_t)seed, (uint32_t)(seed >> 32));
    cudaError_t e = cudaErrorInvalidValue;
    launch_begin("k_quantize_pack_dense", stream);
#define OGQ_LAUNCH_D(SS)                                                                                     \
    e = launch_pdl(k_quantize_pack_dense<SS>, g.ctas, kThreads, 0, stream, d_grad, d_off, T, total, g.chunk, d_levels, \
                   keys, stream_id, d_packed_off, d_packed, quant_steps())
    switch (s) {
        case 3: OGQ_LAUNCH_D(3); break;
        case 5: OGQ_LAUNCH_D(5); break;
        case 9: OGQ_LAUNCH_D(9); break;
        case 17: OGQ_LAUNCH_D(17); break;
        default: return cudaErrorInvalidValue;
    }
#undef OGQ_LAUNCH_D
    launch_end(stream);
    return e;
}

cudaError_t launch_unpack_sum_dense(const uint32_t* const* d_packed_k, const float* const* d_levels_k, int K,
                                    const int64_t* d_off, const int64_t* d_packed_off, int T, int64_t total, int s,
                                    float scale, float* d_out, int sm_count, cudaStream_t stream)
{
    const FlatGrid g = make_flat_grid(total, sm_count * kStreamCtas, 4096);
    cudaError_t e = cudaErrorInvalidValue;
    launch_begin("k_unpack_sum_dense", stream);
    auto bytes = [&](int digits, int row) { return (size_t)(kWarps * 32 * digits + (kWarps + 2) * K * row) * sizeof(float); };
    // shared memory of which four CTAs fit an SM
    constexpr size_t kFour = 54 * 1024;
    auto launch = [&](auto levels, auto digits, auto rest) {
        constexpr int S = decltype(levels)::value, D = decltype(digits)::value, R = decltype(rest)::value;
        e = launch_pdl_smem(k_unpack_sum_dense<S, D, R>, g.ctas, kThreads, bytes(Dense<S>::M, DenseRow<S, D>::kFloats), stream,
                            d_packed_k, d_levels_k, K, d_off, d_packed_off, T, total, g.chunk, scale, d_out);
    };
    auto pick = [&](auto levels, auto digits) {
        constexpr int B = kDenseBatch<decltype(levels)::value>;
        const int rest = K % B;
        if (rest == 0) launch(levels, digits, std::integral_constant<int, 0>{});
        else if (rest == 1) launch(levels, digits, std::integral_constant<int, 1>{});
        else if constexpr (B > 2) {
            if (rest == 2) launch(levels, digits, std::integral_constant<int, 2>{});
            else launch(levels, digits, std::integral_constant<int, 3>{});
        }
    };
    constexpr std::integral_constant<int, 1> one{};
    constexpr std::integral_constant<int, 2> two{};
    constexpr std::integral_constant<int, 3> three{};
    constexpr std::integral_constant<int, 5> five{};
    switch (s) {
        case 3:
            if (bytes(Dense<3>::M, DenseRow<3, 3>::kFloats) <= kFour) pick(three, three);
            else if (bytes(Dense<3>::M, DenseRow<3, 2>::kFloats) <= kFour) pick(three, two);
            else pick(three, one);
            break;
        case 5:
            if (bytes(Dense<5>::M, DenseRow<5, 2>::kFloats) <= kFour) pick(five, two);
            else pick(five, one);
            break;
        case 9: pick(std::integral_constant<int, 9>{}, one); break;
        case 17: pick(std::integral_constant<int, 17>{}, one); break;
        default: return cudaErrorInvalidValue;
    }
    launch_end(stream);
    return e;
}

}  // namespace ogq

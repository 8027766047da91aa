// Fixed-length bucket mode: the gradient is cut into buckets of d elements and every bucket is
// quantized on its own (the setting of all the paper's experiments, d = 128 ... 32768).
//
// One team of threads (a warp for buckets of up to 512 elements, a CTA for longer ones) takes one
// bucket at a time and does the whole path on it: the bucket's values are sorted in shared memory, the
// levels follow from the definitions applied to the sorted values (Algorithm 1 with Q* for ORQ,
// optionally followed by refinement sweeps; the sign change of g for BinGrad-pb; the conditional means
// for BinGrad-b), then the values are quantized and packed.  Results are those of the per-tensor entry
// points called with tensor offsets j * d: same level definitions, same Philox counters (tensor index =
// bucket index), same packed layout.
#include <math.h>

#include <atomic>

#include "ogq_common.cuh"
#include "ogq_internal.h"
#include "ogq_quant.cuh"
#include "ogq_sort.cuh"

namespace ogq {

constexpr int kBktWarpD = 512;         // buckets up to this length are worked on by one warp each
constexpr int kBktWarpsPerCta = 4;     // ... this many to a CTA, independent of one another
constexpr int kBktPrefixMaxD = 4096;   // buckets up to this length keep the prefix sum of every sorted value,
                                       // longer ones that of every thread's first value

struct BktArgs {
    const float* grad;
    int64_t total;
    int d, nb, scheme, s, iters;  // iters: refinement sweeps (ORQ) or Lloyd updates (BinGrad-b)
    float clip_c;                 // > 0: clip every bucket to c times its standard deviation first
    uint32_t stream_id;
    float* levels;
    float* thresh;
    int32_t* status;
    uint32_t* packed;
    int64_t words_per_bucket;
    QuantSteps steps;
};

// Shared memory of one team besides the sort's: level records and the quantizer's table.
struct BktShared {
    SortedLevel lv[kSortedLevels];
    float2 tab[kMaxLevels];  // see quant_table_entry
    int plain;               // the table does not scale
};

// The whole path on bucket j.  EXACT: the bucket fills the team, KPT values for every thread (every full
// bucket whose length is a power of two); otherwise positions are compared with the bucket's length.
template <int BITS, int KPT, bool WARP, bool FULL, bool EXACT>
__device__ __forceinline__ void bkt_encode_one(const BktArgs& A, const PhiloxKeys& pk, int j, int next_j, int len, unsigned char* mem,
                                               BktShared& S, TeamScratch<WARP>& X)
{
    constexpr bool kKeep = KPT <= 16;  // the thread's values stay in registers from the load to the quantizer
    const int lane = threadIdx.x & 31;
    const int t = WARP ? lane : (int)threadIdx.x, nt = WARP ? 32 : (int)blockDim.x;
    const int tw = WARP ? 0 : (int)(threadIdx.x >> 5), ntw = nt >> 5;  // warp inside the team
    const int s = A.s;
    const bool orq = A.scheme == OGQ_ORQ, pbs = A.scheme == OGQ_BINGRAD_PB, threshold = A.scheme == OGQ_BINGRAD_B;
    const int nl = orq ? s : 2;
    float* sv = reinterpret_cast<float*>(mem);
    uint32_t* cells = reinterpret_cast<uint32_t*>(mem);
    double* pre = reinterpret_cast<double*>(mem + (size_t)nt * (KPT + (KPT >= 8 ? 4 : 0)) * sizeof(float));
    const uint32_t tabaddr = (uint32_t)__cvta_generic_to_shared(S.tab);
    {
        const float* src = A.grad + (int64_t)j * A.d;
        const int n = EXACT ? KPT * nt : len;
        int stbits = 0;
        // x / n: of a full bucket, whose length is a power of two, by an exact product.  This and the sums for clipping in a loop of their
        // own are for teams of up to 256 threads (d = 2048, clipped: 171 -> 167 us); in larger ones they cost registers
        // (one bucket of 16384: 20.1 instead of 19.0).  Buckets of other lengths are 2 to 4 % slower with the loop apart when they are
        // clipped and up to 8 % faster when not (25 M elements at d = 640: three levels 268 -> 279, BinGrad-b unclipped 118 -> 109).
        auto over_n = [&](double x) -> double { return EXACT && FULL ? x * (1.0 / (double)KPT) * (WARP ? 0.03125 : __hiloint2double((1023 - (31 - __clz(nt))) << 20, 0)) : x / (double)n; };
        // Element 4 u + c of thread t is value 4 (u nt + t) + c of the bucket: 128-bit loads, all issued
        // before the first use, and the arrangement the quantizer works in.
        auto index = [&](int e) -> int { return 4 * ((e >> 2) * nt + t) + (e & 3); };
        auto have = [&](int e) -> bool { return EXACT || index(e) < n; };
        auto load4 = [&](int u) -> float4 {
            const int i = index(4 * u);
            if (EXACT || i + 3 < n) return __ldg(reinterpret_cast<const float4*>(src + i));
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i < n) v.x = __ldg(src + i);
            if (i + 1 < n) v.y = __ldg(src + i + 1);
            if (i + 2 < n) v.z = __ldg(src + i + 2);
            return v;
        };
        float raw[kKeep ? KPT : 1] = {};
        if constexpr (kKeep) {
#pragma unroll
            for (int u = 0; u < KPT / 4; ++u) {
                const float4 v = load4(u);
                raw[4 * u] = v.x; raw[4 * u + 1] = v.y; raw[4 * u + 2] = v.z; raw[4 * u + 3] = v.w;
            }
        }
        // the next bucket of this team: asked of L2 now
        if (t == 0 && next_j < A.nb - 1) prefetch_l2(A.grad + (int64_t)next_j * A.d, (uint32_t)A.d * 4u);
        auto value = [&](int e) -> float {
            if constexpr (kKeep) return raw[e];
            else return __ldg(src + (have(e) ? index(e) : 0));
        };

        // magnitudes: largest (also tells non-finite values), mean of the leading bits; variance if clipping
        float tau = __int_as_float(0x7f800000);
        uint32_t maxbits = 0u, meanbits = 0u;
        {
            const double v0 = A.clip_c > 0.f ? (double)__ldg(src) : 0.0;
            double sums[2] = {0.0, 0.0};
#pragma unroll
            for (int e = 0; e < KPT; ++e) {
                if (have(e)) {
                    const uint32_t m = __float_as_uint(value(e)) & 0x7fffffffu;
                    maxbits = max(maxbits, m);
                    if (e % 4 == 0) meanbits += m >> 16;
                    if (!FULL && A.clip_c > 0.f) {
                        const double dv = (double)value(e) - v0;
                        sums[0] += dv;
                        sums[1] += dv * dv;
                    }
                }
            }
            if (FULL && A.clip_c > 0.f) {
#pragma unroll
                for (int e = 0; e < KPT; ++e) {
                    if (have(e)) {
                        const double dv = (double)value(e) - v0;
                        sums[0] += dv;
                        sums[1] += dv * dv;
                    }
                }
            }
            team_max_sum<WARP>(maxbits, meanbits, X.u);
            meanbits = (uint32_t)((float)meanbits / (float)((n + 3) >> 2));  // of every fourth value
            if (A.clip_c > 0.f) {
                team_sum<WARP>(sums, X.d);
                double var = over_n(sums[1] - over_n(sums[0] * sums[0]));
                if (!(var > 0.0)) var = 0.0;  // also a non-finite bucket: everything clips to 0
                tau = (float)((double)A.clip_c * sqrt(var));
            }
        }
        const bool bad = maxbits >= 0x7f800000u;
        if (bad) stbits |= OGQ_ST_NONFINITE;
        // clipped, and -0 as 0 (no clipping: tau = +Inf, which also turns a NaN into an infinity)
        auto clip = [&](float x) -> float { return copysignf(fminf(fabsf(x), tau), x) + 0.0f; };
        if constexpr (kKeep) {
            if (A.clip_c > 0.f || bad) {
#pragma unroll
                for (int e = 0; e < KPT; ++e) raw[e] = clip(raw[e]);
            } else {
#pragma unroll
                for (int e = 0; e < KPT; ++e) raw[e] += 0.0f;
            }
        }
        auto clipped = [&](int e) -> float {
            if constexpr (kKeep) return raw[e];
            else return clip(value(e));
        };
        float b0 = 0.f;

        if (threshold) {
            // ---- BinGrad-b: b_0 = mean, b_{-1}, b_1 = conditional means, optional Lloyd updates
            double sum[1] = {0.0};
#pragma unroll
            for (int e = 0; e < KPT; ++e)
                if (have(e)) sum[0] += (double)clipped(e);
            team_sum<WARP>(sum, X.d);
            b0 = (float)over_n(sum[0]);
            long long prev_lo = -1;
            float l_lo = 0.f, l_hi = 0.f;
            for (int it = 0;; ++it) {
                double sp[2] = {0.0, 0.0};
                uint32_t cnt = 0u, none = 0u;
#pragma unroll
                for (int e = 0; e < KPT; ++e) {
                    if (have(e)) {
                        const float v = clipped(e);
                        const bool below = v < b0;
                        sp[0] += below ? (double)v : 0.0;
                        sp[1] += below ? 0.0 : (double)v;
                        cnt += below ? 1u : 0u;
                    }
                }
                team_sum<WARP>(sp, X.d);
                team_max_sum<WARP>(none, cnt, X.u);
                const long long n_lo = (long long)cnt, n_hi = (long long)n - n_lo;
                if (n_lo == 0 || n_hi == 0) {
                    const double m = (n_lo == 0) ? sp[1] / (double)n_hi : sp[0] / (double)n_lo;
                    l_lo = l_hi = (float)m;
                    stbits |= OGQ_ST_CONSTANT;
                    break;
                }
                const double m_lo = sp[0] / (double)n_lo, m_hi = sp[1] / (double)n_hi;
                l_lo = (float)m_lo;
                l_hi = (float)m_hi;
                if (n_lo == prev_lo) break;
                if (it >= A.iters) {
                    if (A.iters > 0) stbits |= OGQ_ST_ITER_CAP;
                    break;
                }
                prev_lo = n_lo;
                b0 = (float)((m_lo + m_hi) * 0.5);
            }
            if (t == 0) {
                A.levels[2 * (int64_t)j] = l_lo;
                A.levels[2 * (int64_t)j + 1] = l_hi;
                A.thresh[j] = b0;
                A.status[j] = stbits;
            }
        } else {
            team_sync<WARP>();  // the previous bucket's levels and table have been read
            if (t == 0) S.plain = 0;
            if (bad) {
                if (t < nl) S.lv[t].v = 0.f;
            } else {
                float r[KPT];
                auto fetch = [&](int e) -> float {
                    const float v = clipped(e);
                    return pbs ? fabsf(v) : v;
                };
                const MagnitudeCells cell(meanbits, fminf(__uint_as_float(maxbits), tau), !pbs,
                                          (uint32_t)(nt * kSortCellsPerThread<KPT>));
                team_sort<KPT, WARP>(r, sv, cells, X.edge, X.u, n, fetch, have, [&](int e) { return cell(fetch(e)); });
                Sorted<KPT, FULL> B;
                B.sv = sv; B.pre = pre; B.n = n;
                {
                    double ls = 0.0, tot;
#pragma unroll
                    for (int e = 0; e < KPT; ++e)
                        if (t * KPT + e < n) ls += (double)r[e];
                    const double base = team_excl_scan<WARP>(ls, X.d, tot);
                    sorted_prefix<KPT, FULL>(r, pre, t, base);
                    if (t == nt - 1 && n == KPT * nt) pre[FULL ? sorted_pre_at<KPT>(n) : nt] = tot;
                }
                team_sync<WARP>();
                if (orq) {
                    if (B.at(0) == B.at(n - 1)) stbits |= OGQ_ST_CONSTANT;
                    if (tw == 0) sorted_orq_levels(B, S.lv, s, A.iters);
                } else if (tw == 0) {
                    const double tot = B.before(n);
                    if (!(tot > 0.0)) stbits |= OGQ_ST_CONSTANT;
                    const float b1 = tot > 0.0 ? sorted_pb_level(B, tot) : 0.f;
                    if (lane < 2) S.lv[lane].v = lane == 0 ? -b1 : b1;
                }
            }
            team_sync<WARP>();
            if (t < nl) {
                const float cur = S.lv[t].v;
                const float nxt = t + 1 < nl ? S.lv[t + 1].v : cur;
                S.tab[t] = quant_table_entry(cur, nxt);
                if (!quant_table_scales(cur, nxt)) S.plain = 1;
                A.levels[(int64_t)j * nl + t] = cur;
            }
            if (t == 0) A.status[j] = stbits;
            team_sync<WARP>();
        }

        // ---- quantize + pack: 128 consecutive elements per warp and trip
        uint32_t* out = A.packed + (int64_t)j * A.words_per_bucket;
        const int region4 = ((n * BITS + 31) / 32 + 3) / 4 * 4;
        const int ngroups = (n + 127) >> 7;
        const float mid = threshold ? 0.f : S.tab[(BITS >= 2) ? (1 << (BITS - 2)) : 0].x;
        const PhiloxHoist hz = philox_hoist(0u, (uint32_t)j, A.stream_id, pk);
        auto group = [&](int g, float4 v) {
            if constexpr (!kKeep) { v.x = clip(v.x); v.y = clip(v.y); v.z = clip(v.z); v.w = clip(v.w); }
            uint32_t bits4;
            if (threshold) {
                bits4 = ((v.x >= b0) ? 1u : 0u) | ((v.y >= b0) ? 2u : 0u) | ((v.z >= b0) ? 4u : 0u) | ((v.w >= b0) ? 8u : 0u);
            } else {
                const uint4 rnd = philox4x32_10_tail(((uint32_t)g << 5) + (uint32_t)lane, hz, pk);
                if (S.plain) {
                    auto level = [&](int k) { return S.lv[k].v; };
                    bits4 = code_as_written<BITS>(v.x, rnd.x, level) | code_as_written<BITS>(v.y, rnd.y, level) << BITS |
                            code_as_written<BITS>(v.z, rnd.z, level) << (2 * BITS) | code_as_written<BITS>(v.w, rnd.w, level) << (3 * BITS);
                } else bits4 = codes_of_entries<BITS>(entry_after_rounding<BITS>(v.x, rnd.x, tabaddr, mid, A.steps),
                                               entry_after_rounding<BITS>(v.y, rnd.y, tabaddr, mid, A.steps),
                                               entry_after_rounding<BITS>(v.z, rnd.z, tabaddr, mid, A.steps),
                                               entry_after_rounding<BITS>(v.w, rnd.w, tabaddr, mid, A.steps), tabaddr);
            }
            const int left = n - ((g << 7) + 4 * lane);  // elements of this lane inside the bucket
            if (!EXACT && left < 4) bits4 &= left > 0 ? (1u << (left * BITS)) - 1u : 0u;
            if constexpr (EXACT) {
                store_chunks<BITS>(out + g * (4 * BITS), bits4, lane);
            } else {
                const uint32_t word = assemble_words<BITS>(bits4, lane);
                const int w = g * (4 * BITS) + packed_word<BITS>(lane);
                if (packs_word<BITS>(lane) && w < region4) out[w] = word;
            }
        };
        if constexpr (kKeep) {
            // (rolled: the unrolled groups' instructions were too many for the instruction cache)
            constexpr int kSide = KPT >= 8 ? 2 : 1;  // groups side by side
#pragma unroll 1
            for (int u = 0; u * ntw + tw < ngroups; u += kSide) {
#pragma unroll
                for (int q = 0; q < kSide; ++q)
                    if (EXACT || (u + q) * ntw + tw < ngroups)
                        group((u + q) * ntw + tw, make_float4(raw[4 * q], raw[4 * q + 1], raw[4 * q + 2], raw[4 * q + 3]));
#pragma unroll
                for (int e = 0; e + 4 * kSide < KPT; ++e) raw[e] = raw[e + 4 * kSide];
            }
        } else {
            for (int u = 0; u * ntw + tw < ngroups; ++u) group(u * ntw + tw, load4(u));
        }
    }
}

template <int BITS, int KPT, bool WARP, bool FULL, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) k_bucket_encode(BktArgs A, size_t team_bytes, const __grid_constant__ PhiloxKeys pk)
{
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int kTeams = WARP ? kBktWarpsPerCta : 1;
    __shared__ BktShared sh_team[kTeams];
    __shared__ TeamScratch<WARP> scratch;
    pdl_wait();
    pdl_launch_dependents();
    const int team = WARP ? (int)(threadIdx.x >> 5) : 0;
    const int P = KPT * (WARP ? 32 : (int)blockDim.x);
    const int step = (int)gridDim.x * kTeams;
    for (int j = (int)blockIdx.x * kTeams + team; j < A.nb; j += step) {
        const int64_t left = A.total - (int64_t)j * A.d;
        const int n = left < (int64_t)A.d ? (int)left : A.d;
        unsigned char* mem = smem + (size_t)team * team_bytes;
        if (n == P) bkt_encode_one<BITS, KPT, WARP, FULL, true>(A, pk, j, j + step, n, mem, sh_team[team], scratch);
        else bkt_encode_one<BITS, KPT, WARP, FULL, false>(A, pk, j, j + step, n, mem, sh_team[team], scratch);
    }
}

static int bkt_pow2(int d)
{
    int P = 128;
    while (P < d) P <<= 1;
    return P;
}

// Shared memory of one team: the sorted values and their prefix sums, or the cells they are sorted with.
template <int KPT, bool FULL>
static size_t bkt_team_bytes(int threads)
{
    const size_t P = (size_t)KPT * threads;
    const size_t sorted = (P + (KPT >= 8 ? P / KPT * 4 : 0)) * sizeof(float) +
                          (FULL ? P + P / KPT + 2 : (size_t)threads + 1) * sizeof(double);
    const size_t cells = (size_t)threads * (kSortCellsPerThread<KPT> + 4) * sizeof(uint32_t);
    return ((sorted > cells ? sorted : cells) + 15) / 16 * 16;
}

template <int BITS, int KPT, bool WARP, bool FULL, int MAXT, int MINB>
static cudaError_t bkt_launch(const BktArgs& A, const PhiloxKeys& pk, int sm_count, cudaStream_t stream)
{
    const int team_threads = WARP ? 32 : bkt_pow2(A.d) / KPT;
    const int teams = WARP ? kBktWarpsPerCta : 1;
    const size_t team_bytes = bkt_team_bytes<KPT, FULL>(team_threads);
    const size_t smem = team_bytes * teams;
    auto kernel = k_bucket_encode<BITS, KPT, WARP, FULL, MAXT, MINB>;
    // The dynamic shared-memory limit and the resident CTAs per SM, looked up once per device and size.
    struct Known { std::atomic<int> resident[6]; };
    static Known known[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int slot = 0;
    while ((32 << slot) < team_threads) ++slot;
    int per_sm = (dev >= 0 && dev < 64) ? known[dev].resident[slot].load(std::memory_order_acquire) : 0;
    if (per_sm == 0) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) return e;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, team_threads * teams, smem);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
        if (dev >= 0 && dev < 64) known[dev].resident[slot].store(per_sm, std::memory_order_release);
    }
    int64_t ctas = (int64_t)per_sm * sm_count;
    const int64_t need = ((int64_t)A.nb + teams - 1) / teams;
    if (ctas > need) ctas = need;
    launch_begin("k_bucket_encode", stream);
    e = launch_pdl(kernel, (int)ctas, team_threads * teams, smem, stream, A, team_bytes, pk);
    launch_end(stream);
    return e;
}

// Values per thread: a bucket of up to 512 elements is one warp's (4, 8 or 16 per lane: its barriers are
// warp barriers and the SM works on as many buckets as it has warps), longer ones a CTA's with 16 per
// thread, the longest with 32.
template <int BITS>
static cudaError_t bkt_dispatch(const BktArgs& A, const PhiloxKeys& pk, int sm_count, cudaStream_t stream)
{
    const int P = bkt_pow2(A.d);
    if (P == 128) return bkt_launch<BITS, 4, true, true, 128, 8>(A, pk, sm_count, stream);
    if (P == 256) return bkt_launch<BITS, 8, true, true, 128, 8>(A, pk, sm_count, stream);
    if (P <= kBktWarpD) return bkt_launch<BITS, 16, true, true, 128, 5>(A, pk, sm_count, stream);
    if (P <= kBktPrefixMaxD) return bkt_launch<BITS, 16, false, true, 256, 3>(A, pk, sm_count, stream);
    if (P == 8192) return bkt_launch<BITS, 16, false, false, 512, 2>(A, pk, sm_count, stream);
    if (P == 16384) return bkt_launch<BITS, 16, false, false, 1024, 1>(A, pk, sm_count, stream);
    return bkt_launch<BITS, 32, false, false, 1024, 1>(A, pk, sm_count, stream);
}

cudaError_t launch_bucket_encode(const float* d_grad, int64_t total, int d, int scheme, int s, int iters,
                                 float clip_c, uint64_t seed, uint32_t stream_id, float* d_levels, float* d_thresh,
                                 int32_t* d_status, uint32_t* d_packed, int sm_count, cudaStream_t stream)
{
    BktArgs A;
    A.grad = d_grad; A.total = total; A.d = d; A.nb = (int)((total + d - 1) / d);
    A.scheme = scheme; A.s = s; A.iters = iters; A.clip_c = clip_c; A.stream_id = stream_id;
    A.levels = d_levels; A.thresh = d_thresh; A.status = d_status; A.packed = d_packed;
    const int bits = ogq_bits_for_levels(s);
    A.words_per_bucket = (int64_t)d * bits / 32;
    A.steps = quant_steps();
    const PhiloxKeys pk = philox_round_keys((uint32_t)seed, (uint32_t)(seed >> 32));
    switch (bits) {
        case 1: return bkt_dispatch<1>(A, pk, sm_count, stream);
        case 2: return bkt_dispatch<2>(A, pk, sm_count, stream);
        case 3: return bkt_dispatch<3>(A, pk, sm_count, stream);
        case 4: return bkt_dispatch<4>(A, pk, sm_count, stream);
        case 5: return bkt_dispatch<5>(A, pk, sm_count, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace ogq

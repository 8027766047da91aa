// Sorting and order statistics of a few hundred to 32768 values on one warp or one CTA, shared by the
// fixed-length buckets and the small tensors of the selection solvers.
#pragma once

#include "ogq_common.cuh"

namespace ogq {

constexpr int kTeamMaxWarps = 32;

// ---------------------------------------------------------------------------
// Teams: a warp (WARP) or the whole CTA.
// ---------------------------------------------------------------------------
template <bool WARP>
__device__ __forceinline__ void team_sync()
{
    if constexpr (WARP) __syncwarp();
    else __syncthreads();
}

// Sums of N doubles over the team, in a fixed order, valid in every thread.  scratch: N * kTeamMaxWarps
// doubles (CTA teams only).
template <bool WARP, int N>
__device__ __forceinline__ void team_sum(double (&v)[N], double* scratch)
{
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = warp_sum(v[i]);
    if constexpr (!WARP) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        __syncthreads();
        if (lane == 0)
#pragma unroll
            for (int i = 0; i < N; ++i) scratch[i * kTeamMaxWarps + warp] = v[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = warp_sum(lane < nw ? scratch[i * kTeamMaxWarps + lane] : 0.0);
    }
}

// Maximum of a and sum of b over the team, valid in every thread.
template <bool WARP>
__device__ __forceinline__ void team_max_sum(uint32_t& a, uint32_t& b, uint32_t* scratch)
{
    a = __reduce_max_sync(0xffffffffu, a);
    b = __reduce_add_sync(0xffffffffu, b);
    if constexpr (!WARP) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        __syncthreads();
        if (lane == 0) { scratch[warp] = a; scratch[kTeamMaxWarps + warp] = b; }
        __syncthreads();
        a = __reduce_max_sync(0xffffffffu, lane < nw ? scratch[lane] : 0u);
        b = __reduce_add_sync(0xffffffffu, lane < nw ? scratch[kTeamMaxWarps + lane] : 0u);
    }
}

// Exclusive sum of v over the team's threads (warps in order); total over the team in tot.
template <bool WARP, class Tv>
__device__ __forceinline__ Tv team_excl_scan(Tv v, Tv* scratch, Tv& tot)
{
    const int lane = threadIdx.x & 31;
    Tv inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const Tv nb = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc = nb + inc;
    }
    const Tv up = __shfl_up_sync(0xffffffffu, inc, 1);
    const Tv own = lane == 0 ? (Tv)0 : up;
    if constexpr (WARP) {
        tot = __shfl_sync(0xffffffffu, inc, 31);
        return own;
    } else {
        const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        __syncthreads();
        if (lane == 31) scratch[warp] = inc;
        __syncthreads();
        Tv w = lane < nw ? scratch[lane] : (Tv)0;
        Tv winc = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const Tv nb = __shfl_up_sync(0xffffffffu, winc, o);
            if (lane >= o) winc = nb + winc;
        }
        tot = __shfl_sync(0xffffffffu, winc, 31);
        const Tv wbase = __shfl_sync(0xffffffffu, winc, warp > 0 ? warp - 1 : 0);
        return warp > 0 ? wbase + own : own;
    }
}

// ---------------------------------------------------------------------------
// Sorting
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cmp_exchange(float& a, float& b)
{
    const float lo = fminf(a, b), hi = fmaxf(a, b);
    a = lo;
    b = hi;
}

// Batcher's odd-even merge sort of a thread's N registers, written out at compile time (N = 16: 63
// compare-exchanges).
template <int N>
__device__ __forceinline__ void sort_thread(float (&r)[N])
{
#pragma unroll
    for (int p = 1; p < N; p <<= 1) {
#pragma unroll
        for (int k = p; k >= 1; k >>= 1) {
#pragma unroll
            for (int i = 0; i + k < N; ++i)
                if (i >= k % p && ((i - k % p) / k) % 2 == 0 && i / (2 * p) == (i + k) / (2 * p)) cmp_exchange(r[i], r[i + k]);
        }
    }
}

// Exchange with thread t ^ m: this thread's register e against the partner's register e (REV false)
// or KPT - 1 - e (REV true); the thread on the lower side keeps the smaller values.
template <int KPT, bool REV>
__device__ __forceinline__ void sort_cross(float (&r)[KPT], float* xch, int m, bool keep_min)
{
    const int t = threadIdx.x, nt = blockDim.x;
    float o[KPT];
    if (m < 32) {
#pragma unroll
        for (int e = 0; e < KPT; ++e) o[e] = __shfl_xor_sync(0xffffffffu, r[REV ? KPT - 1 - e : e], m);
    } else {
        __syncthreads();
#pragma unroll
        for (int e = 0; e < KPT; ++e) xch[e * nt + t] = r[e];
        __syncthreads();
#pragma unroll
        for (int e = 0; e < KPT; ++e) o[e] = xch[(REV ? KPT - 1 - e : e) * nt + (t ^ m)];
    }
#pragma unroll
    for (int e = 0; e < KPT; ++e) r[e] = keep_min ? fminf(r[e], o[e]) : fmaxf(r[e], o[e]);
}

// Ascending bitonic sort of the KPT * (team threads) values held in registers, thread t owning positions
// t * KPT ... of the sequence.  Merges start with a "flip" (position i against i ^ (k - 1)) followed by
// halvings (i against i ^ j), so every compare-exchange puts the smaller value at the lower position.
// Only buckets whose values the cells of team_sort cannot separate come here.  xch: one float per position
// (CTA teams only).
template <int KPT, bool WARP>
__device__ __noinline__ void sort_bitonic(float (&r)[KPT], float* xch)
{
    const int t = WARP ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
    const int P = KPT * (WARP ? 32 : (int)blockDim.x);
    sort_thread<KPT>(r);
    for (int k = 2 * KPT; k <= P; k <<= 1) {
        const int m = k / KPT - 1;
        sort_cross<KPT, true>(r, xch, m, (t & ((m + 1) >> 1)) == 0);
        for (int j = k >> 2; j >= KPT; j >>= 1) sort_cross<KPT, false>(r, xch, j / KPT, (t & (j / KPT)) == 0);
#pragma unroll
        for (int j = KPT / 2; j >= 1; j >>= 1) {
#pragma unroll
            for (int e = 0; e < KPT; ++e)
                if ((e & j) == 0) cmp_exchange(r[e], r[e | j]);
        }
    }
    if constexpr (!WARP) __syncthreads();
}

// Index of sorted position i in shared memory: four words of padding after every thread's KPT values, so
// that the 128-bit accesses of neighbouring threads fall into different banks.
template <int KPT>
__device__ __forceinline__ int sorted_at(int i)
{
    return KPT >= 8 ? i + i / KPT * 4 : i;
}
// The same for the fp64 prefix sums (one double of padding).
template <int KPT>
__device__ __forceinline__ int sorted_pre_at(int i)
{
    return i + i / KPT;
}

// Cells per thread of the sort.  Two to four cells per value where shared memory allows it.
template <int KPT>
constexpr int kSortCellsPerThread = KPT <= 8 ? 16 : 32;

// The cells of values that may lie anywhere: a monotone map that spreads the usual gradient distributions
// (one peak around 0, tails of any weight) almost evenly over nc cells.  The cell of v is given by the
// leading bits of the float 1 + k |v|, which are a piecewise linear log2, with k = 2 / (geometric mean of
// the magnitudes), scaled so that the largest magnitude falls into the last cell, negative values mirrored.
// Zeros get a cell of their own and so do the values of the largest magnitude (all the clipped ones): those
// two values may be there in any number, and equal values need no order among themselves.
struct MagnitudeCells {
    float k;
    uint32_t range, mul, base;

    // mean_bits: mean of (magnitude bits >> 16), maxabs: largest magnitude, signed_values: false when all
    // values are magnitudes (BinGrad-pb)
    __device__ __forceinline__ MagnitudeCells(uint32_t mean_bits, float maxabs, bool signed_values, uint32_t nc)
    {
        float geo = __uint_as_float(mean_bits << 16);
        geo = fmaxf(geo, fmaxf(maxabs * 0x1p-20f, 1e-37f));
        k = __fdividef(2.0f, geo);
        range = __float_as_uint(fmaf(maxabs, k, 1.0f)) - 0x3f800000u;
        const uint32_t side = signed_values ? nc / 2 : nc;
        base = signed_values ? nc / 2 : 0u;
        // floor((side - 2) * 2^32 / (range + 1)), a little less: umulhi(x, mul) < side - 2 for every x <= range
        mul = range > 2 * side ? (uint32_t)((float)(side - 2) * 0.99999f * (4294967296.0f / ((float)range + 1.0f))) : 0u;
    }
    __device__ __forceinline__ uint32_t operator()(float v) const
    {
        const uint32_t x = __float_as_uint(fmaf(fabsf(v), k, 1.0f)) - 0x3f800000u;
        return base + ((__umulhi(x, mul) + min(x, 1u) + (x == range ? 1u : 0u)) ^ (uint32_t)((int)__float_as_uint(v) >> 31));
    }
};

// Sorts the team's n values into sv (position i at sorted_at<KPT>(i); positions n .. P hold +Inf) and leaves
// thread t the KPT values at positions t * KPT ... in r.  fetch(e) returns the e-th of the thread's own
// values (any arrangement), have(e) whether there is one, cell_of(e) its cell, a monotone function of it
// below kSortCellsPerThread<KPT> times the number of threads.
//
// A counting sort into the cells, then a repair of the order inside the cells.  The counts are added up
// over the cells in order and every value goes to the next free position of its cell.  Each value is then
// at most a cell's width from its place, and a few passes of odd-even transposition (KPT - 1 exchanges in
// registers, one with the next thread) put it there; a comparison of all neighbours tells when.  Values
// that the cells do not separate (a narrow peak far from 0) are left to the bitonic network after
// kRepairs rounds.
//   What bounds it: instruction issue on the integer / min-max pipe.  About 25 instructions per value,
// whatever the length, against 60 (one warp) to 130 (32 warps, plus their exchanges through shared
// memory) of the bitonic network that did the whole sort before: with it the bucket encoder's launch for
// 25.6 M values, ORQ s = 9, took 351 us at d = 512, 384 at 2048, 694 at 32768; now 153, 168 and 242.
//   cells: shared memory for the cells (four words of padding to every thread's); sv may lie over it.
template <int KPT, bool WARP, class Fetch, class Have, class CellOf>
__device__ __forceinline__ void team_sort(float (&r)[KPT], float* sv, uint32_t* cells, float* edge, uint32_t* scan_scratch,
                                          int n, Fetch fetch, Have have, CellOf cell_of)
{
    constexpr int CPT = kSortCellsPerThread<KPT>;
    constexpr int kPasses = 3, kRepairs = 3;
    const int lane = threadIdx.x & 31;
    const int t = WARP ? lane : (int)threadIdx.x, nt = WARP ? 32 : (int)blockDim.x;
    const int P = KPT * nt;

    uint4* mine = reinterpret_cast<uint4*>(cells + t * (CPT + 4));
#pragma unroll
    for (int q = 0; q < CPT / 4; ++q) mine[q] = make_uint4(0u, 0u, 0u, 0u);
    team_sync<WARP>();
    uint32_t at[KPT];  // where the counter of the value's cell is
#pragma unroll
    for (int e = 0; e < KPT; ++e) {
        at[e] = 0u;
        if (have(e)) {
            const uint32_t c = cell_of(e);
            at[e] = c + c / CPT * 4;
            atomicAdd(cells + at[e], 1u);
        }
    }
    team_sync<WARP>();
    {
        // exclusive sums over the cells, in place: this thread's CPT consecutive ones
        uint32_t sum = 0u;
#pragma unroll
        for (int q = 0; q < CPT / 4; ++q) {
            const uint4 w = mine[q];
            sum += (w.x + w.y) + (w.z + w.w);
        }
        uint32_t tot;
        uint32_t run = team_excl_scan<WARP>(sum, scan_scratch, tot);
#pragma unroll
        for (int q = 0; q < CPT / 4; ++q) {
            const uint4 w = mine[q];
            uint4 o;
            o.x = run; o.y = o.x + w.x; o.z = o.y + w.y; o.w = o.z + w.z;
            run = o.w + w.w;
            mine[q] = o;
        }
    }
    team_sync<WARP>();
    // the next free position of the value's cell
#pragma unroll
    for (int e = 0; e < KPT; ++e)
        if (have(e)) at[e] = atomicAdd(cells + at[e], 1u);
    team_sync<WARP>();  // the cells are dead: sv may lie over them
#pragma unroll
    for (int e = 0; e < KPT; ++e)
        if (have(e)) sv[sorted_at<KPT>((int)at[e])] = fetch(e);
    for (int i = n + t; i < P; i += nt) sv[sorted_at<KPT>(i)] = __int_as_float(0x7f800000);
    team_sync<WARP>();
    float4* own = reinterpret_cast<float4*>(sv + sorted_at<KPT>(t * KPT));
#pragma unroll
    for (int q = 0; q < KPT / 4; ++q) {
        const float4 w = own[q];
        r[4 * q] = w.x; r[4 * q + 1] = w.y; r[4 * q + 2] = w.z; r[4 * q + 3] = w.w;
    }
    for (int round = 0;; ++round) {
#pragma unroll
        for (int pass = 0; pass < kPasses; ++pass) {
#pragma unroll
            for (int e = 0; e + 1 < KPT; e += 2) cmp_exchange(r[e], r[e + 1]);
#pragma unroll
            for (int e = 1; e + 1 < KPT; e += 2) cmp_exchange(r[e], r[e + 1]);
            // the pair that two threads share
            float nx = __shfl_down_sync(0xffffffffu, r[0], 1), pv = __shfl_up_sync(0xffffffffu, r[KPT - 1], 1);
            if constexpr (WARP) {
                if (lane == 31) nx = r[KPT - 1];
                if (lane == 0) pv = r[0];
            } else {
                const int warp = threadIdx.x >> 5;
                float* ed = edge + (pass & 1) * 2 * kTeamMaxWarps;
                if (lane == 0) ed[2 * warp] = r[0];
                if (lane == 31) ed[2 * warp + 1] = r[KPT - 1];
                __syncthreads();
                if (lane == 31) nx = t + 1 < nt ? ed[2 * warp + 2] : r[KPT - 1];
                if (lane == 0) pv = t > 0 ? ed[2 * warp - 1] : r[0];
            }
            r[KPT - 1] = fminf(r[KPT - 1], nx);
            r[0] = fmaxf(r[0], pv);
        }
        // (the pairs that two threads share are in order: the exchange above came last)
        bool ok = true;
#pragma unroll
        for (int e = 0; e + 1 < KPT; ++e) ok = ok && r[e] <= r[e + 1];
        if (WARP ? __all_sync(0xffffffffu, ok) : __syncthreads_and(ok)) break;
        if (round >= kRepairs) {
            float tmp[KPT];
#pragma unroll
            for (int e = 0; e < KPT; ++e) tmp[e] = r[e];
            sort_bitonic<KPT, WARP>(tmp, sv);
#pragma unroll
            for (int e = 0; e < KPT; ++e) r[e] = tmp[e];
            break;
        }
    }
#pragma unroll
    for (int q = 0; q < KPT / 4; ++q) own[q] = make_float4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
    team_sync<WARP>();
}

// ---------------------------------------------------------------------------
// Levels from the sorted values
// ---------------------------------------------------------------------------
struct SortedLevel {
    float v;
    int i_lt, i_le;      // #{values < v}, #{values <= v}
    double s_lt, s_le;   // sums of those
};

// Sorted values of a bucket with prefix sums.  FULL: pre holds the sum before every position, else the
// sum before every thread's first position and the rest is added up from the values.
template <int KPT, bool FULL>
struct Sorted {
    const float* sv;
    const double* pre;
    int n;

    __device__ __forceinline__ float at(int i) const { return sv[sorted_at<KPT>(i)]; }

    __device__ __forceinline__ double before(int i) const
    {
        if constexpr (FULL) {
            return pre[sorted_pre_at<KPT>(i)];
        } else {
            const int t = i / KPT;
            double a = pre[t];
            for (int q = t * KPT; q < i; ++q) a += (double)at(q);
            return a;
        }
    }
    __device__ __forceinline__ int lower(float v, int hi) const  // first position in [0, hi) that holds a value >= v
    {
        int lo = 0;
        while (lo < hi) { const int mid = (lo + hi) >> 1; if (at(mid) < v) lo = mid + 1; else hi = mid; }
        return lo;
    }
    __device__ __forceinline__ int upper(float v, int lo) const  // first position in [lo, n) that holds a value > v
    {
        int hi = n;
        while (lo < hi) { const int mid = (lo + hi) >> 1; if (at(mid) <= v) lo = mid + 1; else hi = mid; }
        return lo;
    }
    // first and last-plus-one position of the run of values equal to at(p) (usually p alone)
    __device__ __forceinline__ int run_begin(int p, float v) const { return (p > 0 && at(p - 1) == v) ? lower(v, p) : p; }
    __device__ __forceinline__ int run_end(int p, float v) const { return (p + 1 < n && at(p + 1) == v) ? upper(v, p + 1) : p + 1; }

    __device__ __forceinline__ SortedLevel level_at(int p) const
    {
        SortedLevel l;
        l.v = at(p);
        l.i_lt = run_begin(p, l.v);
        l.i_le = run_end(p, l.v);
        l.s_lt = before(l.i_lt);
        l.s_le = FULL ? before(l.i_le) : l.s_lt + (double)l.v * (double)(l.i_le - l.i_lt);
        return l;
    }
    // Q*(L, R), R > L: with T = sum_{L <= v <= R} (v - L) / (R - L) the position of the (floor(T) + 1)-th largest value of the
    // segment.  (Of L only i_lt and s_lt are used, of R only i_le and s_le.)
    __device__ __forceinline__ int qstar_at(const SortedLevel& L, const SortedLevel& R) const
    {
        const double Lv = (double)L.v, Rv = (double)R.v;
        const int m = R.i_le - L.i_lt;
        const double A = (R.s_le - L.s_lt) - Lv * (double)m;
        const int k = __double2int_rd(A / (Rv - Lv));  // floor
        return R.i_le - 1 - min(max(k, 0), m - 1);
    }
    __device__ __forceinline__ SortedLevel qstar(const SortedLevel& L, const SortedLevel& R) const
    {
        if (!(R.v > L.v)) return L;
        return level_at(qstar_at(L, R));
    }
};

constexpr int kSortedLevels = 17;  // most levels of a tensor or bucket

// ORQ levels of sorted values, by the 32 lanes of one warp: Algorithm 1, a level after its two brackets, the
// levels of one depth on as many lanes; then up to `sweeps` refinement sweeps (every interior level again
// from its two current neighbours, ascending).  lv: s records in shared memory.
//   What is not used is not worked out: the end levels are only ever the lower (the upper) bracket, and the levels of the last depth
// nobody's unless there are sweeps.  (The searches for the end levels' runs of equal values, which clipping makes long, and the last
// depth's sums took 24 of 179 us for 25.6 M clipped values at d = 512, s = 9, and 3 to 5 % without clipping.)
template <int KPT, bool FULL>
__device__ __forceinline__ void sorted_orq_levels(const Sorted<KPT, FULL>& B, SortedLevel* lv, int s, int sweeps)
{
    const int lane = threadIdx.x & 31;
    if (lane < 2) {
        SortedLevel l;  // (both ends' fields, of which lv[0] needs the lower ones and lv[s - 1] the upper ones)
        l.v = B.at(lane == 0 ? 0 : B.n - 1);
        l.i_lt = 0;
        l.i_le = B.n;
        l.s_lt = 0.0;
        l.s_le = B.before(B.n);
        lv[lane == 0 ? 0 : s - 1] = l;
    }
    __syncwarp();
#pragma unroll 1
    for (int stride = (s - 1) >> 1; stride >= (sweeps > 0 ? 1 : 2); stride >>= 1) {
        const int q = stride + lane * 2 * stride;
        if (q < s - 1) lv[q] = B.qstar(lv[q - stride], lv[q + stride]);
        __syncwarp();
    }
    if (sweeps <= 0) {
        const int q = 1 + 2 * lane;
        if (q < s - 1) {
            const SortedLevel &L = lv[q - 1], &R = lv[q + 1];
            lv[q].v = R.v > L.v ? B.at(B.qstar_at(L, R)) : L.v;
        }
        __syncwarp();
    }
    if (lane == 0) {
        for (int it = 0; it < sweeps; ++it) {
            bool changed = false;
            for (int q = 1; q < s - 1; ++q) {
                const SortedLevel l = B.qstar(lv[q - 1], lv[q + 1]);
                if (l.v != lv[q].v) { lv[q] = l; changed = true; }
            }
            if (!changed) break;
        }
    }
}

// The BinGrad-pb level b_1 of sorted magnitudes with a positive sum `tot`, by the 32 lanes of one warp: the
// last magnitude x_c with g(x_c) = x_c n - sum_{|v| >= x_c} |v| <= 0 is found (g does not decrease along
// the sorted magnitudes; 32 candidates are tried at a time), the sign change lies in [x_c, next magnitude).
template <int KPT, bool FULL>
__device__ __forceinline__ float sorted_pb_level(const Sorted<KPT, FULL>& B, double tot)
{
    const int lane = threadIdx.x & 31;
    const double n = (double)B.n;
    int lo = 0, hi = B.n;  // the answer lies in [lo, hi) (position 0 when g is positive everywhere)
    while (hi - lo > 1) {
        const int step = (hi - lo + 31) >> 5;
        const int i = lo + lane * step;
        bool below = false;
        if (i < hi) {
            const float x = B.at(i);
            below = (double)x * n - (tot - B.before(B.run_begin(i, x))) <= 0.0;
        }
        const unsigned m = __ballot_sync(0xffffffffu, below);
        const int k = m ? 31 - __clz(m) : 0;
        lo += k * step;
        hi = (lo + step < hi) ? lo + step : hi;
    }
    const float x = B.at(lo);
    const double stat_up = (tot - B.before(B.run_end(lo, x))) / n;
    return (float)(stat_up > (double)x ? stat_up : (double)x);
}

// Scratch of a CTA team's block-wide sums and scans, and of the pairs its warps share in the sort.
template <bool WARP>
struct TeamScratch {
    double d[WARP ? 1 : 3 * kTeamMaxWarps];
    uint32_t u[WARP ? 1 : 2 * kTeamMaxWarps];
    float edge[WARP ? 1 : 4 * kTeamMaxWarps];
};

// Thread t's part of the prefix sums; base: the sum before its first value.
template <int KPT, bool FULL>
__device__ __forceinline__ void sorted_prefix(const float (&r)[KPT], double* pre, int t, double base)
{
    if constexpr (FULL) {
        double run = base;
        double* p = pre + sorted_pre_at<KPT>(t * KPT);
#pragma unroll
        for (int e = 0; e < KPT; ++e) {
            p[e] = run;
            run += (double)r[e];  // +Inf past the end: those positions are never asked for
        }
    } else {
        pre[t] = base;
    }
}

}  // namespace ogq

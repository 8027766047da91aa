// ORQ and BinGrad-pb level solvers: exact selection by histogram refinement.
//
// Round 1 streams the bucket once: per tensor it finds min, max and a histogram
// over key cells (128 cells per binade inside a 16-binade window anchored at a
// sampled magnitude, one cell per binade outside), each cell with an exact
// count and an exact integer sum of the low key bits.  A launch with one CTA
// per tensor then solves on the cell prefix sums and leaves a few narrow
// candidate intervals.  Round 2 streams the bucket again, against round 1's
// direction, and copies the few percent of elements inside the intervals to scratch.  What follows depends on their
// number:
//   up to kSortN            round 2 only copies them; one CTA indexes the copied keys and finishes the tensor.
//   ORQ, more, and room     round 2 copies them in order of round 1's cells; every level is selected among the keys of the
//                           cell that holds its rank, by one CTA, or where a cell has many, by a cluster (k_sel_round3).
//   otherwise               round 2 counts them on a finer grid as well; another launch per tensor solves again, and round
//                           3 and later work on the copied keys only, until every level's rank falls into a single-key
//                           cell or one CTA's index holds the rest.
// Tensors of at most kSmallN elements are not streamed: the second solver launch indexes them in shared memory.  The key
// buffers hold one eighth of the bucket: a pass whose copies do not fit is repeated on the gradient with
// the narrower intervals.
//
// All cross-CTA accumulation is integer (atomic adds, min, max), and a rank does not depend on the order in which
// values reach their cells: counts are exact, sums of what one cell holds are exact but for values of many
// binades, and an integer T is recognised within their rounding (floor_of_t).  No kernel waits on another CTA but for the
// clusters of round 3; the slices of a tensor there are counted off by an atomic, and the last CTA goes on with the solver.
//   What bounds it: the rounds stream at 4.7 to 5.1 TB/s from DRAM, bound by the integer pipe and the wait for their loads
// (60 % of the issue slots); the solver launches are bound by the latency of one CTA's barriers and of code that runs once
// (ResNet-50 bucket, nine levels: about 13 and 16 of 135 us, 20,000 and 30,000 cycles).  Running them on made-up cells
// while they wait, so that their instructions are in the cache, gained nothing: the second run takes as long as the first.
// Solving in the streaming kernels, by the CTA that arrived last, took 89 and 125 us for the two rounds of that bucket
// instead of 61 and 61.
#include <math.h>

#include <stddef.h>

#include <algorithm>
#include <atomic>

#include "ogq_common.cuh"
#include "ogq_internal.h"
#include "ogq_select_solver.cuh"
#include "ogq_sort.cuh"
#include "ogq_ws.h"

namespace ogq {

constexpr int kSelThreads = 512;    // two CTAs are resident per SM: a CTA in a solver pass, a sort or a
                                    // set-up phase leaves the other half of the SM streaming
constexpr int kSelResident = 2;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSolveThreads = 1024;  // of the solver launches
constexpr int kSelW = 16;          // binades in the fine window of round 1
constexpr int kSelM = 7;           // log2(cells per binade) in the window
constexpr int kSmallN = 16384;     // tensors up to this size are solved in shared memory
constexpr int kSortN = 16384;      // candidates from which one CTA finishes a larger tensor
constexpr int kStageCap = 320;     // per-warp staging entries for compaction
constexpr int kMaxSlices = 64;     // CTAs that share one tensor's copied keys in round 3
constexpr int kSliceElems = 16384;
constexpr int kMaxRounds = 32;
constexpr int kScanMax = 16384, kScanMaxAlone = 65536;  // longest list of copied keys one CTA looks through for the last few
                                                        // thousand (the second where no other kernel would do it)
constexpr int kRefineMax = 32;     // runs of candidate cells that make up the intervals of the next round

constexpr int kRound1Mag = 256 - kSelW + (kSelW << kSelM);  // round-1 cells per sign
constexpr int kRound1Cells = 2 * kRound1Mag;
static_assert(kRound1Cells <= kCells, "round-1 cells exceed the budget");

// TState::compact_only: what the next pass does with the keys inside the intervals.
constexpr int kCounted = 0;        // copies them and counts them on finer cells
constexpr int kCompact = 1;        // copies them: they fit one CTA's index
constexpr int kOrdered = 2;        // copies them in order of round 1's cells; the second solver launch selects among one cell's at a time
constexpr int kOrderedLarger = 3;  // the same, with cells so large that round 3 does it, with a cluster of CTAs

struct TState {
    int done, round, m, hi_e;
    unsigned kmin_inv, kmax, nonfinite;
    unsigned arrive;    // slices that have arrived in round 3; of a tensor copied in order of round 1's cells, the keys of the fullest
    unsigned expected;  // CTAs that work on the tensor in round 3; the candidate cells of a tensor copied in their order
    int compact_only;
    int overflow;      // the current pass dropped copies that did not fit the tensor's region
    int from_grad;     // the current pass (round >= 3) reads the gradient, not the previous pass's copies
    unsigned long long cursor[2];
    long long n;
    long long cand;  // elements inside the intervals
    double stot;
    Interval iv[kMaxIv];
    ExactLv lv[kMaxLv];
};

struct SelWs {
    TState* st;                  // [T]
    uint32_t* gcnt;              // [T][kCells]
    unsigned long long* glsum;   // [T][kCells]
    unsigned* nitems;            // [2] work items of round 3
    int2* items;                 // [T * kMaxSlices], from the end on: tensors copied in order of their cells (nitems[1] of them)
    uint32_t* buf[2];            // [total / kBufDiv] copied keys: tensor t owns [sel_region(off[t]), sel_region(off[t+1]))
};

// The copied keys of a tensor are normally a few percent of it, so the two key buffers hold one eighth
// of the bucket: the tensor that starts at element x owns the words from sel_region(x) on, up to where
// the next tensor's region starts.  A pass whose copies do not fit drops the surplus and marks the
// tensor (TState::overflow); the next pass then reads the gradient again instead of the buffer, with
// narrower intervals, until the copies fit.
constexpr int kBufDiv = 8;
__host__ __device__ __forceinline__ int64_t sel_region(int64_t x) { return (x / kBufDiv) & ~(int64_t)3; }

static size_t sel_zero_bytes(int T)
{
    return align_up(sizeof(TState) * (size_t)T, 256) + align_up(sizeof(uint32_t) * (size_t)T * kCells, 256) +
           align_up(sizeof(unsigned long long) * (size_t)T * kCells, 256) + 256;
}

size_t ws_bytes_select(int T, int64_t total, int /*s*/)
{
    return sel_zero_bytes(T) + align_up(sizeof(int2) * (size_t)T * kMaxSlices, 256) +
           2 * align_up(sizeof(uint32_t) * (size_t)(total / kBufDiv + 8), 256);
}

static SelWs sel_carve(void* base, int T, int64_t total)
{
    char* p = (char*)base;
    SelWs w;
    w.st = (TState*)p; p += align_up(sizeof(TState) * (size_t)T, 256);
    w.gcnt = (uint32_t*)p; p += align_up(sizeof(uint32_t) * (size_t)T * kCells, 256);
    w.glsum = (unsigned long long*)p; p += align_up(sizeof(unsigned long long) * (size_t)T * kCells, 256);
    w.nitems = (unsigned*)p; p += 256;
    w.items = (int2*)p; p += align_up(sizeof(int2) * (size_t)T * kMaxSlices, 256);
    w.buf[0] = (uint32_t*)p; p += align_up(sizeof(uint32_t) * (size_t)(total / kBufDiv + 8), 256);
    w.buf[1] = (uint32_t*)p;
    return w;
}

// ---------------------------------------------------------------------------
// Shared-memory layout of a streaming CTA (dynamic): cell counters, low-bit sums
// (two 32-bit halves with carry), and the per-warp compaction stages.  The
// solver reuses the same bytes for its prefix arrays.
// ---------------------------------------------------------------------------
constexpr size_t kSmemHist = 3 * kCells * sizeof(uint32_t);
constexpr size_t kSmemStage = kSelWarps * kStageCap * sizeof(uint32_t);

// Every structure in shared memory that a function which is not inlined uses lies in the dynamic shared memory and is reached
// through this symbol: through a reference it would be read by generic loads.
extern __shared__ __align__(16) unsigned char smem[];

// A candidate cell of round 1 of a tensor whose keys are copied in order of these cells; the table lies where the tensor's finer
// cells would have their sums, the cursors of the cells where they would have their counts.
constexpr int kCandCells = 512;  // at most
constexpr int kCellBits = 23;    // log2 of the keys of the widest cell
// Most keys of a cell that the second solver launch selects among by itself, and most where round 3 has other tensors to work on anyway (which then
// takes no longer).  One tensor of 6 M elements, nine levels: 109 -> 90 us; the VGG-19 bucket, with the first limit alone: 496 -> 517.
constexpr int kCellsAlone = 16384, kCellsBeside = 4096;
static_assert(kCandCells <= 1 << (32 - kCellBits), "a cell's number fits above its keys");
struct CandCell {
    double sbefore;      // sum of the elements below it
    uint32_t cbefore, n; // number of these, and of its own
    uint32_t klo, base;  // lowest key; where its own begin in the tensor's region (a multiple of four)
    int sh, pad;         // log2 of the keys
};
static_assert(sizeof(CandCell) * kCandCells <= sizeof(unsigned long long) * kCells, "the table fits");

struct Round2Ctx {  // per-CTA constants of round 2, kept in shared memory to spare registers
    uint32_t* dst;
    unsigned long long* cursor;
    uint32_t clear;  // 0x7fffffff when only magnitudes count
    int mode;        // TState::compact_only: whether, and in what order, keys are copied without counting them
    uint32_t* cursors;       // of the candidate cells
    unsigned long long cap;  // words of the tensor's region in the destination buffer
    int* overflow;           // set when a copy did not fit
};

struct Table {  // interval lookup table of the tensor being streamed
    uint32_t klo[kMaxIv];
    uint32_t khi[kMaxIv];
    int sh[kMaxIv];
    int cellbase[kMaxIv];
    int m, ncells;
    int lo_e;                                      // bottom binade of the round-1 fine window
    uint32_t coarse[1024];                         // one bit per block of 2^17 keys that touches an interval
    Round2Ctx ctx;
    int fills[kSolveThreads / 32];                 // values parked per warp
    int cta_fill;                                  // mode 2: keys in the CTA's buffer
};
// Mode 2 counts nothing: in place of the cells lie, for every candidate cell, where its keys begin and this CTA's number of
// them (then their place), and the CTA's buffer.
struct Partition {
    uint32_t base[kCandCells], cnt[kCandCells];
    uint32_t buffer[kSmemHist / sizeof(uint32_t) - 2 * kCandCells];
};
constexpr int kCtaBuffer = (int)(kSmemHist / sizeof(uint32_t)) - 2 * kCandCells;
__device__ __forceinline__ Partition& sel_partition() { return *reinterpret_cast<Partition*>(smem); }
// the cells, the table, the stages (of the streaming kernels' sixteen warps, or of round 3's 32)
constexpr size_t kOffStage = kSmemHist + (sizeof(Table) + 15) / 16 * 16;
constexpr size_t kStreamBytes = kOffStage + kSmemStage;
__device__ __forceinline__ Table& sel_table() { return *reinterpret_cast<Table*>(smem + kSmemHist); }
__device__ __forceinline__ uint32_t* sel_hist() { return reinterpret_cast<uint32_t*>(smem); }
__device__ __forceinline__ uint32_t* sel_stage() { return reinterpret_cast<uint32_t*>(smem + kOffStage); }

// By the first kMaxIv threads of the CTA (called by all threads; the caller synchronises afterwards).
__device__ __forceinline__ void table_from_intervals(Table& tb, const Interval* iv, int m)
{
    const int j = threadIdx.x;
    if (j < kMaxIv) {
        if (j < m) {
            tb.klo[j] = iv[j].klo; tb.khi[j] = iv[j].khi; tb.sh[j] = iv[j].sh; tb.cellbase[j] = iv[j].cellbase;
        } else {
            tb.klo[j] = 0xffffffffu; tb.khi[j] = 0u; tb.sh[j] = 0; tb.cellbase[j] = 0;
        }
    }
    if (j == 0) {
        tb.m = m;
        tb.ncells = (m > 0) ? iv[m - 1].cellbase + iv[m - 1].ncell : 0;
    }
}

// Round-1 interval j of the layout: coarse (one cell per binade) outside a window of kSelW binades that ends
// at binade hi_e, fine inside; six of them, in key order, or the three of the non-negative values only.
// (One of them may have no cells.)
__device__ __forceinline__ Interval round1_interval(int hi_e, bool magnitude_only, int j)
{
    const int lo_e = hi_e - kSelW;
    if (magnitude_only) j += 3;
    // cells of the coarse part below the window, of the window and of the part above it, mirrored for negative values
    const int part = j < 3 ? 2 - j : j - 3;
    const int ncell = part == 0 ? lo_e : part == 1 ? (kSelW << kSelM) : 256 - hi_e;
    const int before = part == 0 ? 0 : part == 1 ? lo_e : lo_e + (kSelW << kSelM);  // cells nearer to zero
    const int edge = part == 0 ? 0 : part == 1 ? lo_e : hi_e;                        // lowest binade
    const int width = part == 1 ? kSelW : ncell;                                     // in binades
    Interval x;
    x.sh = part == 1 ? 23 - kSelM : 23;
    x.ncell = ncell;
    x.klo = j < 3 ? 0x80000000u - ((uint32_t)(edge + width) << 23) : 0x80000000u + ((uint32_t)edge << 23);
    x.khi = x.klo + (uint32_t)((((unsigned long long)ncell) << x.sh) - 1ull);
    x.cellbase = magnitude_only ? before : j < 3 ? kRound1Mag - before - ncell : kRound1Mag + before;
    x.pad = 0;
    x.cbefore = 0;
    x.sbefore = 0.0;
    return x;
}

// A pass that only copies keys writes them as interval (top bits) and distance from its lowest key, so that the finish need not
// search for the interval again (it took 18,000 of 40,000 cycles for 14,000 keys): intervals of at most 2^kRelBits keys.
constexpr int kRelBits = 26;
static_assert(kMaxIv <= 1 << (32 - kRelBits), "an interval's number fits the top bits");

__device__ __forceinline__ bool classify(const Table& tb, uint32_t key, int& cell, uint32_t& low, int& sh, uint32_t& packed)
{
    int idx = 0;
#pragma unroll
    for (int step = kMaxIv / 2; step >= 1; step >>= 1)
        if (tb.klo[idx + step] <= key) idx += step;
    sh = tb.sh[idx];
    const uint32_t rel = key - tb.klo[idx];
    packed = (uint32_t)idx << kRelBits | (rel & ((1u << kRelBits) - 1u));
    cell = tb.cellbase[idx] + (int)(rel >> sh);
    low = rel & ((1u << sh) - 1u);
    return key >= tb.klo[idx] && key <= tb.khi[idx];
}

__device__ __forceinline__ void hist_add(uint32_t* cnt, uint32_t* lo, uint32_t* hi, int cell, uint32_t low)
{
    atomicAdd(cnt + cell, 1u);
    if (low) {
        const uint32_t old = atomicAdd(lo + cell, low);
        if (old + low < old) atomicAdd(hi + cell, 1u);
    }
}

// Warp-uniform visit of base[pb, pe): every lane of a warp calls f(x, nvalid) the same number of
// times (nvalid = 0, 1 or 4), so f may use warp collectives.  128-bit loads on the aligned body.
__device__ __forceinline__ uint4 ld4(const uint4* p) { return __ldcg(p); }
__device__ __forceinline__ uint32_t ld1(const uint32_t* p) { return __ldcg(p); }

template <class E4, class E, class F>
__device__ __forceinline__ void warp_visit4(const E* __restrict__ base, int64_t pb, int64_t pe, F f)
{
    int64_t a = (pb + 3) & ~(int64_t)3;
    if (a > pe) a = pe;
    int64_t b = pe & ~(int64_t)3;
    if (b < a) b = a;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nt = blockDim.x;
    if (warp == 0) {
        E x[4];
        int nv = 0;
        if (lane < (int)(a - pb)) { x[0] = ld1(base + pb + lane); nv = 1; }
        else if (lane >= 4 && lane - 4 < (int)(pe - b)) { x[0] = ld1(base + b + lane - 4); nv = 1; }
        f(x, nv);
    }
    const E4* b4 = reinterpret_cast<const E4*>(base);
    const int64_t e = b >> 2;
    for (int64_t i0 = (a >> 2) + warp * 32; i0 < e; i0 += 4 * nt) {
        E x[4][4];
        int nx[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t i = i0 + (int64_t)u * nt + lane;
            nx[u] = 0;
            if (i < e) {
                const E4 v = ld4(b4 + i);
                x[u][0] = v.x; x[u][1] = v.y; x[u][2] = v.z; x[u][3] = v.w;
                nx[u] = 4;
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i0 + (int64_t)u * nt < e) f(x[u], nx[u]);
    }
}

struct Stager {  // per-warp compaction stage
    uint32_t* stage;            // this warp's kStageCap entries in shared memory
    uint32_t* dst;              // tensor's region in the destination buffer
    unsigned long long* cursor; // tensor's append cursor
    int fill;

    __device__ __forceinline__ void flush()
    {
        const int lane = threadIdx.x & 31;
        if (fill > 0) {
            unsigned long long pos = 0;
            if (lane == 0) pos = atomicAdd(cursor, (unsigned long long)fill);
            pos = __shfl_sync(0xffffffffu, pos, 0);
            for (int i = lane; i < fill; i += 32) dst[pos + i] = stage[i];
        }
        __syncwarp();
        fill = 0;
    }

    // every lane passes its own keys (c of them, c <= 4)
    __device__ __forceinline__ void append(const uint32_t* kk, int c)
    {
        const int lane = threadIdx.x & 31;
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int nb = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += nb;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        if (total == 0) return;
        const int at = fill + incl - c;
        for (int i = 0; i < c; ++i) stage[at + i] = kk[i];
        fill += total;
        __syncwarp();
        if (fill > kStageCap - 128) flush();
    }
};

__device__ __forceinline__ float min3f(float a, float b, float c)
{
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));  // a NaN operand is skipped
    return r;
}
__device__ __forceinline__ float max3f(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
constexpr int kPrefetchTrips = 2;                         // how far ahead of the loads L2 is asked for a block
constexpr uint32_t kTripBytes = 4u * kSelThreads * 16u;  // one trip of a CTA's streaming loop
// shared-memory add without a return value, on a 32-bit shared address
__device__ __forceinline__ void red_shared_add(uint32_t addr, uint32_t v)
{
    asm volatile("red.shared.add.u32 [%0], %1;" :: "r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t atom_shared_add(uint32_t addr, uint32_t v)
{
    uint32_t old;
    asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(addr), "r"(v) : "memory");
    return old;
}

constexpr int kPackedPerSign = kSelW << kSelM;  // fine cells per sign (2048)
constexpr int kPackedCells = 2 * kPackedPerSign;
// Loop trips between two folds of the packed cells, in which no cell should take 256 values: of magnitudes a normal distribution has
// 0.38 % in one cell, a uniform one 0.39 % (round 1 of 120 M normal magnitudes: 200 us with eight trips, most of them done again, 97 with six).
template <bool MAG>
constexpr int kPackTrips = MAG ? 6 : 8;
static_assert(kPackedCells * sizeof(uint32_t) <= kSelWarps * kStageCap * sizeof(uint32_t),
              "the packed cells live in the (otherwise unused) compaction stages during round 1");

template <bool MAG, bool CLIP>
struct Round1Body {
    uint32_t lo23;
    uint32_t neg_lo23x2;  // -(lo23 << 1), the addend of the doubled window offset
    int lo_e;
    uint32_t cnt;  // shared address of the count of the first non-negative magnitude cell; the low
                   // sums lie kCells words above the counts, their carries 2 kCells words above
    uint32_t pk;   // shared address of the packed words: kPackedPerSign cells of the non-negative values,
                   // then (signed keys only) kPackedPerSign cells of the negative ones, both by magnitude
    uint32_t coarse;  // shared address of the counter of values that bypassed the packed cells
    uint32_t one24;   // 1 << 24 (the count field of a packed word), kept in a register
    float mn, mx;
    uint32_t nonfinite;
    float tau;         // clipping threshold (CLIP only)
    float tau_mag;     // its magnitude: that of a clipped value, also where a caller's threshold is negative
    uint32_t clipped;  // values at that magnitude since the last fold; of those, the negative ones in the upper half (CLIP only)

    // clip to [-tau, tau] (CLIP), magnitude for BinGrad-pb, and fold -0 into +0
    __device__ __forceinline__ float canon(float v) const
    {
        if (CLIP) {
            const float m = fminf(fabsf(v), tau);
            return (MAG ? m : copysignf(m, v)) + 0.0f;
        }
        return (MAG ? fabsf(v) : v) + 0.0f;
    }

    // A value inside the fine window, the slow way: two adds into the wide counters (cells and low bits
    // mirrored for negative values, so that both ascend with the key).  rel = magnitude bits - lo23.
    __device__ __forceinline__ void fine_wide(uint32_t bits, uint32_t rel)
    {
        const int sgn = MAG ? 0 : ((int)bits >> 31);  // 0 or -1
        const uint32_t low = (bits ^ (uint32_t)sgn) & ((1u << (23 - kSelM)) - 1u);
        const uint32_t c = cnt + (uint32_t)(((lo_e + (int)(rel >> (23 - kSelM))) ^ sgn) << 2);
        red_shared_add(c, 1u);
        const uint32_t old = atom_shared_add(c + 4u * kCells, low);
        if (old + low < old) red_shared_add(c + 8u * kCells, 1u);
    }

    // The fast way: one shared-memory add of {count 1 in the top 8 bits, low magnitude bits in the other
    // 24} into the cell's packed word (r2 = rel << 1, below kSelW << 24).  The caller folds the packed
    // words into the wide counters every few trips, before a cell can have taken 256 values (and redoes
    // the trips the slow way if one did); the mirroring of the negative half happens there.  The
    // instruction mix matters here: the loop is bound by the integer/logic pipe, so the address is put
    // together with multiply-adds and the sign is not branched on.
    __device__ __forceinline__ void fine_packed(uint32_t bits, uint32_t r2)
    {
        // pk + 4 * cell, cell = r2 >> (24 - kSelM): the high half of a multiply-add by a power of two,
        // which the compiler turns into one shift-and-add
        static_assert(kSelM == 7, "the shift below is 32 - (24 - kSelM - 2)");
        uint32_t addr;
        asm("mad.hi.u32 %0, %1, 131072, %2;" : "=r"(addr) : "r"(r2 & ~((1u << (24 - kSelM)) - 1u)), "r"(pk));
        if (!MAG) asm("mad.lo.u32 %0, %1, %2, %0;" : "+r"(addr) : "r"(bits >> 31), "r"(4u * kPackedPerSign));
        const uint32_t word = (bits & ((1u << (23 - kSelM)) - 1u)) | one24;
        if constexpr (CLIP) {
            uint32_t count = 1u;
            if (!MAG) asm("mad.lo.u32 %0, %1, 65536, %2;" : "=r"(count) : "r"(bits >> 31), "r"(one24 >> 24));
            // (unordered: a threshold that is not a number clips nothing, see canon)
            asm volatile("{ .reg .pred p; setp.ltu.f32 p, %3, %4; @p red.shared.add.u32 [%1], %2; @!p add.u32 %0, %0, %5; }"
                         : "+r"(clipped) : "r"(addr), "r"(word), "f"(fabsf(__uint_as_float(bits))), "f"(tau_mag), "r"(count) : "memory");
        } else {
            red_shared_add(addr, word);
        }
    }

    // any value (already canonical)
    template <bool PACKED>
    __device__ __forceinline__ void any(uint32_t bits)
    {
        const int sgn = MAG ? 0 : ((int)bits >> 31);
        const uint32_t mag = bits & 0x7fffffffu;
        const uint32_t rel = mag - lo23;
        if (rel < ((uint32_t)kSelW << 23)) {
            if (PACKED) fine_packed(bits, rel << 1);  // (counts a clipped value aside)
            else fine_wide(bits, rel);
        } else {  // outside the fine window: one cell per binade
            const int e = (int)(mag >> 23);
            const int mi = (e < lo_e) ? e : e - kSelW + (kSelW << kSelM);
            if (e == 255) nonfinite = 1u;  // the window never reaches binade 255
            const uint32_t c = cnt + (uint32_t)((mi ^ sgn) << 2);
            const uint32_t low = (mag ^ (uint32_t)sgn) & 0x7fffffu;
            red_shared_add(c, 1u);
            const uint32_t old = atom_shared_add(c + 4u * kCells, low);
            if (old + low < old) red_shared_add(c + 8u * kCells, 1u);
            if (PACKED) red_shared_add(coarse, 1u);
        }
    }

    __device__ __forceinline__ void one(float v)
    {
        v = canon(v);
        mn = fminf(mn, v);
        mx = fmaxf(mx, v);
        any<false>(__float_as_uint(v));
    }

    template <bool PACKED>
    __device__ __forceinline__ void four(float4 x)
    {
        const float v0 = canon(x.x), v1 = canon(x.y), v2 = canon(x.z), v3 = canon(x.w);
        mn = min3f(min3f(mn, v0, v1), v2, v3);
        mx = max3f(max3f(mx, v0, v1), v2, v3);
        const uint32_t b0 = __float_as_uint(v0), b1 = __float_as_uint(v1), b2 = __float_as_uint(v2),
                       b3 = __float_as_uint(v3);
        // doubled offset into the window, (magnitude bits - lo23) << 1: the doubling drops the sign bit,
        // and a multiply-add does both steps outside the integer/logic pipe
        uint32_t r0, r1, r2, r3;
        asm("mad.lo.u32 %0, %1, 2, %2;" : "=r"(r0) : "r"(b0), "r"(neg_lo23x2));
        asm("mad.lo.u32 %0, %1, 2, %2;" : "=r"(r1) : "r"(b1), "r"(neg_lo23x2));
        asm("mad.lo.u32 %0, %1, 2, %2;" : "=r"(r2) : "r"(b2), "r"(neg_lo23x2));
        asm("mad.lo.u32 %0, %1, 2, %2;" : "=r"(r3) : "r"(b3), "r"(neg_lo23x2));
        // the window spans kSelW = 2^4 binades, so "all four inside" is one test on the OR (a value
        // below the window wraps to at least kSelW << 24 as well, because lo23 < 2^31 - 2^27)
        static_assert((kSelW & (kSelW - 1)) == 0, "window size must be a power of two");
        if ((r0 | r1 | r2 | r3) < ((uint32_t)kSelW << 24)) {
            if (PACKED) {
                fine_packed(b0, r0); fine_packed(b1, r1); fine_packed(b2, r2); fine_packed(b3, r3);
            } else {
                fine_wide(b0, r0 >> 1); fine_wide(b1, r1 >> 1); fine_wide(b2, r2 >> 1); fine_wide(b3, r3 >> 1);
            }
        } else {
            any<PACKED>(b0); any<PACKED>(b1); any<PACKED>(b2); any<PACKED>(b3);
        }
    }
};

// Round 1 over grad[pb, pe): per element min / max and the cell histogram (count, sum of the low key
// bits).  The bulk goes through packed cells (one shared-memory add per element instead of two, see
// Round1Body::fine), folded into the wide counters every kPackTrips loop trips; the sum of the folded
// counts is checked against the number of values that went in, and a mismatch (a cell took 256 values
// or more within the trips: heavily repeated values) redoes those trips with the two-add path.
// The packed cells (the compaction stages) are zero before, and zero again on return.
struct Round1Out {
    float vmin, vmax;
    uint32_t nonfinite;
};

template <bool MAG, bool CLIP>
__device__ __noinline__ Round1Out stream_round1(const float* __restrict__ grad, int64_t pb, int64_t pe, int lo_e, float tau)
{
    __shared__ uint32_t sh_coarse, sh_total, sh_clipped[2];
    uint32_t *hist = sel_hist(), *packed = sel_stage();
    Round1Body<MAG, CLIP> f;
    f.tau = tau;
    f.tau_mag = fabsf(tau);
    f.lo23 = (uint32_t)lo_e << 23;
    f.neg_lo23x2 = 0u - (f.lo23 << 1);
    f.one24 = 0x01000000u;
    f.lo_e = lo_e;
    f.cnt = (uint32_t)__cvta_generic_to_shared(hist + (MAG ? 0 : kRound1Mag));
    f.pk = (uint32_t)__cvta_generic_to_shared(packed);
    f.coarse = (uint32_t)__cvta_generic_to_shared(&sh_coarse);
    f.mn = __int_as_float(0x7f800000); f.mx = __int_as_float(0xff800000); f.nonfinite = 0u;
    f.clipped = 0u;
    if (CLIP && threadIdx.x < 2) sh_clipped[threadIdx.x] = 0u;
    // the body from the first 32-byte boundary on, whole blocks of eight floats
    int64_t a = pb + (int64_t)((0u - (uint32_t)(reinterpret_cast<uintptr_t>(grad + pb) >> 2)) & 7u);
    if (a > pe) a = pe;
    const int64_t b = a + ((pe - a) & ~(int64_t)7);
    const int tid = threadIdx.x;
    if (tid < (int)(a - pb)) f.one(__ldg(grad + pb + tid));
    if (tid < (int)(pe - b)) f.one(__ldg(grad + b + tid));
    const int ntrips = (int)((b - a) / (16 * kSelThreads));  // full trips: the same for every thread
    constexpr int kNp = MAG ? kPackedPerSign : kPackedCells;
    // upwards; downwards behind the clipping threshold's pass, which went up
    constexpr int kStep = CLIP ? -16 * kSelThreads : 16 * kSelThreads;
    const float* src = grad + a + 8 * tid + (CLIP ? (int64_t)(ntrips - 1) * 16 * kSelThreads : 0);  // this thread's next load
    int pf_left = ntrips - kPrefetchTrips;
    for (int t0 = 0; t0 < ntrips; t0 += kPackTrips<MAG>) {
        const int nt = min(ntrips - t0, kPackTrips<MAG>);
        if (tid == 0) { sh_coarse = 0u; sh_total = 0u; }
        __syncthreads();
        const float* const period = src;
        for (int tt = 0; tt < nt; ++tt) {
            if (tid == 0 && pf_left > 0) prefetch_l2(src + kPrefetchTrips * kStep, kTripBytes);
            --pf_left;
            float4 x[4];
#pragma unroll
            for (int u = 0; u < 4; u += 2) load8(src + u * 4 * kSelThreads, x[u], x[u + 1]);
            src += kStep;
#pragma unroll
            for (int u = 0; u < 4; ++u) f.template four<true>(x[u]);
        }
        __syncthreads();
        // fold, phase 1: do the packed counts add up to the values that went in?
        uint32_t mine = 0u;
        uint32_t wv[kNp / kSelThreads];  // this thread's packed words, read once
#pragma unroll
        for (int k = 0; k < kNp / kSelThreads; ++k) {
            wv[k] = packed[tid + k * kSelThreads];
            mine += wv[k] >> 24;
        }
        if constexpr (CLIP) {
            const uint32_t all = __reduce_add_sync(0xffffffffu, f.clipped & 0xffffu), neg = MAG ? 0u : __reduce_add_sync(0xffffffffu, f.clipped >> 16);
            mine += f.clipped & 0xffffu;
            f.clipped = 0u;
            if ((tid & 31) == 0) {
                if (all) atomicAdd(&sh_clipped[0], all - neg);
                if (neg) atomicAdd(&sh_clipped[1], neg);
            }
        }
        mine = __reduce_add_sync(0xffffffffu, mine);
        if ((tid & 31) == 0 && mine) atomicAdd(&sh_total, mine);
        __syncthreads();
        const bool ok = sh_total + sh_coarse == (uint32_t)nt * 16u * kSelThreads;
        // phase 2: into the wide counters (packed index p: negative values mirror below the middle)
#pragma unroll
        for (int k = 0; k < kNp / kSelThreads; ++k) {
            const int p = tid + k * kSelThreads;
            const uint32_t w = wv[k];
            if (w) {
                packed[p] = 0u;
                if (ok) {
                    // non-negative half: cell and low bits ascend with the magnitude; negative half: mirrored
                    const uint32_t c = w >> 24, sum = w & 0xffffffu;
                    const bool neg = !MAG && p >= kPackedPerSign;
                    const int cell = MAG ? lo_e + p
                                         : (neg ? kRound1Mag - 1 - lo_e - (p - kPackedPerSign) : kRound1Mag + lo_e + p);
                    hist[cell] += c;
                    const uint32_t add = neg ? c * ((1u << (23 - kSelM)) - 1u) - sum : sum;
                    const uint32_t old = hist[kCells + cell];
                    hist[kCells + cell] = old + add;
                    if (old + add < old) hist[2 * kCells + cell] += 1u;  // carry into the high word
                }
            }
        }
        if (!ok) {
            // a packed count wrapped: the fine values of these trips again, two adds each (the values outside
            // the window were counted directly the first time and are skipped now)
            __syncthreads();
            for (int tt = 0; tt < nt; ++tt) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float4 x = __ldg(reinterpret_cast<const float4*>(period + tt * kStep + (u >> 1) * 8 * kSelThreads) + (u & 1));
                    const float vv[4] = {f.canon(x.x), f.canon(x.y), f.canon(x.z), f.canon(x.w)};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint32_t bits = __float_as_uint(vv[j]);
                        const uint32_t rel = (bits & 0x7fffffffu) - f.lo23;
                        if (rel < ((uint32_t)kSelW << 23) && !(CLIP && fabsf(vv[j]) >= f.tau_mag)) f.fine_wide(bits, rel);
                    }
                }
            }
        }
        __syncthreads();  // everyone has read the totals before they are reset
    }
    __syncthreads();
    const float4* rest = reinterpret_cast<const float4*>(grad + a + (int64_t)ntrips * 16 * kSelThreads);
    for (int i = tid; i < (int)((b - a) / 4) - ntrips * 4 * kSelThreads; i += kSelThreads) f.template four<false>(__ldg(rest + i));
    if constexpr (CLIP) {
        // the clipped values, all of one magnitude: counted aside, because they would wrap the packed count of their cell in every
        // period (three clipped levels of the ResNet-50 bucket: round 1 took 52 us, with every period done again, now 38)
        __syncthreads();
        if (threadIdx.x < 2 && sh_clipped[threadIdx.x]) {
            // (only values inside the fine window are counted aside, so the threshold lies in it)
            const bool neg = threadIdx.x == 1;
            const uint32_t mag = __float_as_uint(f.tau_mag), rel = mag - f.lo23, n = sh_clipped[threadIdx.x];
            const int mi = lo_e + (int)(rel >> (23 - kSelM)), cell = (MAG ? 0 : kRound1Mag) + (neg ? ~mi : mi);
            const uint32_t low = (neg ? ~mag : mag) & ((1u << (23 - kSelM)) - 1u);
            const unsigned long long sum = ((unsigned long long)hist[2 * kCells + cell] << 32 | hist[kCells + cell]) + (unsigned long long)n * low;
            hist[cell] += n;
            hist[kCells + cell] = (uint32_t)sum;
            hist[2 * kCells + cell] = (uint32_t)(sum >> 32);
        }
    }
    return Round1Out{f.mn, f.mx, f.nonfinite};
}

// Round 2 over grad[pb, pe).  Phase A: a one-bit-per-2^17-bit-patterns test on the raw fp32 bits
// rejects almost every element; values that pass are parked in the warp's stage (no classification
// yet).  Phase B, whenever the stage fills up: the parked values are turned into keys and classified
// exactly 32 at a time, so that the expensive part runs with all lanes busy; keys inside an interval
// are histogrammed and copied out.
// A key copied in order of the candidate cells: to position `at` of the tensor's region, as its distance from the cell's lowest key.
__device__ __forceinline__ void partition_store(const Table& tb, uint32_t code, uint32_t at)
{
    if (at < tb.ctx.cap) tb.ctx.dst[at] = code & ((1u << kCellBits) - 1u);
}

// The CTA's buffer to the cells' places, which it reserves with one addition per cell.  Called by every thread.
__device__ __forceinline__ void partition_flush()
{
    Table& tb = sel_table();
    Partition& part = sel_partition();
    __syncthreads();
    const int n = min(tb.cta_fill, kCtaBuffer);
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += blockDim.x) atomicAdd(&part.cnt[part.buffer[i] >> kCellBits], 1u);
    __syncthreads();
    for (int c = threadIdx.x; c < kCandCells; c += blockDim.x)
        if (part.cnt[c]) part.cnt[c] = part.base[c] + atomicAdd(tb.ctx.cursors + c, part.cnt[c]);
    __syncthreads();
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const uint32_t code = part.buffer[i];
        partition_store(tb, code, atomicAdd(&part.cnt[code >> kCellBits], 1u));
    }
}

// Phase B of round 2 for one warp: classifies `fill` parked values 32 at a time.  A free function
// taking values, so that the caller's per-warp state can stay in registers.
__device__ __noinline__ void round2_drain(int fill)
{
    Table* tb = &sel_table();
    const Round2Ctx* ctx = &tb->ctx;
    uint32_t* hist = sel_hist();
    const uint32_t* stage = sel_stage() + (threadIdx.x >> 5) * kStageCap;
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t clear = ctx->clear;
    __syncwarp();
    for (int base = 0; base < fill; base += 32) {
        const int i = base + lane;
        uint32_t key = 0;
        bool in = false;
        if (i < fill) {
            uint32_t bits = stage[i] & clear;
            if (bits == 0x80000000u) bits = 0u;
            key = bits ^ ((uint32_t)((int)bits >> 31) | 0x80000000u);
            int cell, sh;
            uint32_t low, packed;
            in = classify(*tb, key, cell, low, sh, packed);
            if (ctx->mode == 1) key = packed;
            else if (ctx->mode == 2) key = (uint32_t)cell << kCellBits | low;
            else if (in) hist_add(hist, hist + kCells, hist + 2 * kCells, cell, low);
        }
        const uint32_t m2 = __ballot_sync(0xffffffffu, in);
        if (ctx->mode == 2) {
            // into the CTA's buffer; what that does not hold goes to its cell's place at once
            int pos = 0;
            if (lane == 0 && m2) pos = atomicAdd(&tb->cta_fill, __popc(m2));
            pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(m2 & lt);
            Partition& part = sel_partition();
            if (in && pos < kCtaBuffer) part.buffer[pos] = key;
            else if (in) partition_store(*tb, key, part.base[key >> kCellBits] + atomicAdd(ctx->cursors + (key >> kCellBits), 1u));
        } else if (m2) {
            unsigned long long pos = 0;
            if (lane == 0) pos = atomicAdd(ctx->cursor, (unsigned long long)__popc(m2));
            pos = __shfl_sync(0xffffffffu, pos, 0);
            if (in) {
                const unsigned long long at = pos + __popc(m2 & lt);
                if (at < ctx->cap) ctx->dst[at] = key;
                else *(volatile int*)ctx->overflow = 1;
            }
        }
    }
    __syncwarp();
}

// Marks, in the space of raw fp32 bit patterns, every block of 2^17 patterns that can hold a value
// whose key lies in one of the table's intervals (called by all threads).  A block of 2^17 aligned
// keys is a block of 2^17 aligned patterns; -0 shares the block of the smallest negative values, and
// with magnitude_only both signs of a pattern are marked.  Block b of a word sits at bit 31 - (b & 31):
// a left shift by the block index brings its bit to the top of the word.
__device__ __forceinline__ void build_prefilter(Table& tb, bool magnitude_only)
{
    for (int i = threadIdx.x; i < 1024; i += blockDim.x) tb.coarse[i] = 0u;
    __syncthreads();
    if ((int)threadIdx.x < tb.m) {
        const uint32_t ba = tb.klo[threadIdx.x] >> 17, bb = tb.khi[threadIdx.x] >> 17;
        for (uint32_t b = ba; b <= bb; ++b) {
            const uint32_t pblk = (b & 0x4000u) ? (b ^ 0x4000u) : (~b & 0x7fffu);
            atomicOr(&tb.coarse[pblk >> 5], 0x80000000u >> (pblk & 31));
            if (magnitude_only || pblk == 0u) {
                const uint32_t twin = pblk ^ 0x4000u;
                atomicOr(&tb.coarse[twin >> 5], 0x80000000u >> (twin & 31));
            }
        }
    }
    __syncthreads();
}

template <bool CLIP>
struct Round2Warp {
    uint32_t coarse;  // shared addresses: the table's prefilter bitmap,
    uint32_t stage;   // this warp's kStageCap parking slots,
    uint32_t fillp;   // and their fill counter (bumped by the lanes that hit)
    float tau;        // clipping threshold (CLIP only)

    __device__ __forceinline__ float clip(float v) const { return CLIP ? copysignf(fminf(fabsf(v), tau), v) : v; }

    // Phase A for one element: no warp collective, only the lanes that pass the bitmap test do work.
    __device__ __forceinline__ void park(uint32_t bits)
    {
        const uint32_t pos = atom_shared_add(fillp, 1u);
        asm volatile("st.shared.u32 [%0], %1;" :: "r"(stage + (pos << 2)), "r"(bits) : "memory");
    }
    // Word address = coarse + ((bits & ~(2^22 - 1)) >> 20), written as the high half of a multiply-add
    // by 2^12: the compiler makes one shift-and-add of it (a real multiplication, with the factor
    // hidden in a kernel argument, was measured slower).  The funnel shift takes its count modulo 32.
    __device__ __forceinline__ uint32_t top_is_hit(uint32_t bits) const
    {
        uint32_t addr, word;
        asm("mad.hi.u32 %0, %1, 4096, %2;" : "=r"(addr) : "r"(bits & 0xffc00000u), "r"(coarse));
        asm("ld.shared.u32 %0, [%1];" : "=r"(word) : "r"(addr));
        return __funnelshift_l(0u, word, bits >> 17);  // the block's bit is now bit 31
    }
    __device__ __forceinline__ void one(float v)
    {
        const uint32_t bits = __float_as_uint(clip(v));
        if (top_is_hit(bits) >> 31) park(bits);
    }
    // Branch-free form for the main loop: shifts `hits` left and appends this element's bit.
    __device__ __forceinline__ void test(float v, uint32_t& hits) const
    {
        hits = __funnelshift_l(top_is_hit(__float_as_uint(clip(v))), hits, 1);
    }
    // Parks the elements marked in `hits` (bit 15 = the first of the sixteen elements tested: p[0], ..., p[7],
    // p[stride], ..., p[stride + 7]).  The values are read again, from L1: a hit is
    // rare, and a register cannot be picked by a run-time index.
    __device__ __forceinline__ void park_hits(uint32_t hits, const float* p, int stride)
    {
        while (hits) {
            const int b = 31 - __clz(hits);
            hits &= ~(1u << b);
            const int j = 15 - b;
            park(__float_as_uint(clip(__ldg(p + (j >> 3) * stride + (j & 7)))));
        }
    }
};

// NT: threads of the CTA; DOWN: from the end of the piece to its beginning.  The table and its Round2Ctx are complete.
// Inlined: as a function of its own, with what its callers' limits leave it, a pass over 143.7 M elements took 135 us
// instead of 113.
template <bool CLIP, int NT, bool DOWN>
__device__ __forceinline__ void stream_round2(const float* __restrict__ grad, int64_t pb, int64_t pe, float tau)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Table& tb = sel_table();
    int* fills = tb.fills;
    if (lane == 0) fills[warp] = 0;
    __syncwarp();
    Round2Warp<CLIP> w;
    w.tau = tau;
    w.coarse = (uint32_t)__cvta_generic_to_shared(tb.coarse);
    w.stage = (uint32_t)__cvta_generic_to_shared(sel_stage() + warp * kStageCap);
    w.fillp = (uint32_t)__cvta_generic_to_shared(&fills[warp]);
    // the body from the first 32-byte boundary on, whole blocks of eight floats
    int64_t a = pb + (int64_t)((0u - (uint32_t)(reinterpret_cast<uintptr_t>(grad + pb) >> 2)) & 7u);
    if (a > pe) a = pe;
    const int64_t b = a + ((pe - a) & ~(int64_t)7);
    if (warp == 0) {  // ragged head and tail, one element per lane
        if (lane < (int)(a - pb)) w.one(__ldg(grad + pb + lane));
        else if (lane >= 8 && lane - 8 < (int)(pe - b)) w.one(__ldg(grad + b + lane - 8));
        __syncwarp();
    }
    const float* const body = grad + a + 8 * lane;
    const int64_t e = (b - a) >> 3;    // blocks
    int64_t i0 = warp * 32;            // the trip counts below are warp-uniform
    // Trips of 2 x NT blocks (contiguous, 64 NT bytes per CTA).  One thread asks
    // L2 for the block kPrefetchTrips ahead, so that the loads below find their lines there.
    // A lane tests its sixteen values of a trip without branching; the warp then parks the trip's
    // hits in one go (nearly every trip has a hit in some lane, so the divergent parking code is
    // paid once per trip, not once per few values).  `fill` mirrors the stage's fill counter in a
    // register: it is the same in all lanes, so whether to drain first is a uniform decision.
    const int64_t rest = e - i0 - NT - 32;
    const int64_t trips = rest >= 0 ? rest / (2 * NT) + 1 : 0, after = i0 + trips * 2 * NT;
    constexpr int64_t step = DOWN ? -2 * NT : 2 * NT;
    if (DOWN) i0 += (trips - 1) * 2 * NT;
    // blocks to ask for: thread 0's trips, but for one upwards that the CTA's last warps do not have
    int64_t pf_left = trips - kPrefetchTrips - (!DOWN && after > e ? 1 : 0);
    __syncwarp();
    int fill = *(volatile int*)&fills[warp];
    auto park = [&](uint32_t hits, const float* p) {
        for (;;) {  // one turn, unless the stage has to be drained to make room
            const int tot = (int)__reduce_add_sync(0xffffffffu, (uint32_t)__popc(hits));
            if (tot == 0) break;
            if (fill + tot <= kStageCap) {
                if (hits) w.park_hits(hits, p, 8 * NT);
                fill += tot;
                break;
            }
            if (fill) {
                round2_drain(fill);
                if (lane == 0) fills[warp] = 0;
                __syncwarp();
                fill = 0;
                continue;
            }
            // more hits in one trip than the empty stage holds: the first eight values of every lane now
            const uint32_t first = hits & 0xff00u;
            if (first) w.park_hits(first, p, 8 * NT);
            fill = (int)__reduce_add_sync(0xffffffffu, (uint32_t)__popc(first));
            hits &= 0xffu;
        }
    };
    auto last_trip = [&]() {  // the blocks after the whole trips
        if (after >= e) return;
        const float* p = body + 8 * after;
        float4 x[4];
#pragma unroll
        for (int u = 0; u < 4; u += 2) {
            x[u] = x[u + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (after + lane + (u / 2) * NT < e) load8(p + u * 4 * NT, x[u], x[u + 1]);
        }
        uint32_t hits = 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            w.test(x[u].x, hits); w.test(x[u].y, hits); w.test(x[u].z, hits); w.test(x[u].w, hits);
            if (after + lane + (u / 2) * NT >= e) hits &= ~15u;
        }
        park(hits, p);
    };
    if (DOWN) last_trip();
    for (int64_t k = 0; k < trips; ++k, i0 += step) {
        const float* p = body + 8 * i0;
        if (threadIdx.x == 0 && k < pf_left) prefetch_l2(p + kPrefetchTrips * 8 * step, 4u * NT * 16u);
        float4 x[4];
#pragma unroll
        for (int u = 0; u < 4; u += 2) load8(p + u * 4 * NT, x[u], x[u + 1]);
        uint32_t hits = 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            w.test(x[u].x, hits); w.test(x[u].y, hits); w.test(x[u].z, hits); w.test(x[u].w, hits);
        }
        park(hits, p);
    }
    if (!DOWN) last_trip();
    __syncwarp();
    round2_drain(*(volatile int*)&fills[warp]);
}

// Streams copied keys [pb, pe) of a tensor: counts those inside the intervals on the cells and copies them on, or copies them
// on as interval and distance (nohist).
__device__ __forceinline__ void stream_piece(const uint32_t* __restrict__ src, int64_t pb, int64_t pe, const Table& tb,
                                             uint32_t* cnt, uint32_t* lo, uint32_t* hi, Stager& stg, bool nohist)
{
    warp_visit4<uint4, uint32_t>(src, pb, pe, [&](const uint32_t* x, int nv) {
        uint32_t kk[4];
        int c = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j >= nv) continue;
            int cell, sh;
            uint32_t low, packed;
            if (classify(tb, x[j], cell, low, sh, packed)) {
                if (!nohist) hist_add(cnt, lo, hi, cell, low);
                kk[c++] = nohist ? packed : x[j];
            }
        }
        stg.append(kk, c);
    });
}

__device__ __forceinline__ void zero_hist(uint32_t* smem_hist, int ncells)
{
    for (int i = threadIdx.x; i < ncells; i += blockDim.x) {
        smem_hist[i] = 0u;
        smem_hist[kCells + i] = 0u;
        smem_hist[2 * kCells + i] = 0u;
    }
}

__device__ __forceinline__ void flush_hist(const uint32_t* smem_hist, int ncells, uint32_t* gcnt,
                                           unsigned long long* glsum)
{
    for (int i = threadIdx.x; i < ncells; i += blockDim.x) {
        const uint32_t c = smem_hist[i];
        if (c) {
            atomicAdd(gcnt + i, c);
            const unsigned long long l =
                ((unsigned long long)smem_hist[2 * kCells + i] << 32) | smem_hist[kCells + i];
            if (l) atomicAdd(glsum + i, l);
        }
    }
}

// The kernels from here to solver_round work on one tensor with one CTA and run their code once: what they
// spend is the latency of barriers, of dependent loads and of instructions that are not in the instruction
// cache yet.  So loops stay rolled, values live in shared memory instead of unrolled registers, a warp works
// on one level with searches spread over its lanes, and fp64 division is one function.
__device__ __noinline__ double fp64_div(double a, double b) { return a / b; }

struct __align__(16) SolverShared {
    Interval iv[kMaxIv];
    Interval niv[kMaxIv];
    LvInfo lv[kMaxLv];
    SolverView view;
    uint32_t sc[32];
    double ss[32];
    int pb_a, pb_b, pb_c;
    int done, nm, internal, nopen;
    uint32_t offc[kMaxIv];    // per-interval shifts of the scanned prefix arrays
    double offs[kMaxIv];
    uint32_t marks[(kSlots + 31) / 32];  // candidate cells, one bit per slot
    int pa[kRefineMax], pb[kRefineMax];  // runs of candidate cells
    long long cand;           // elements inside the new intervals
    // finish
    uint4 place[kMaxIv];        // of the intervals: lowest and highest key (padded: no key lies in the surplus ones), first cell, log2 of the keys per cell
    uint32_t before[kMaxIv];    // elements of the tensor below the interval (surplus ones: more than there are)
    int start[kMaxIv + 1];      // position of the interval's first value
    double pre[kMaxIv];         // sum of the values before it
    int n_keys;
    uint32_t below[32];
};

__device__ __forceinline__ SolverShared& sel_state();

// Exclusive sums of (c, s) over the CTA's threads in thread order; totals in tot_c, tot_s.  Any number of warps.  (The warps'
// sums are added up by one warp: by all of them for themselves, the shuffles of 32 warps took 3200 cycles in all.)
__device__ __forceinline__ void block_excl_scan(uint32_t& c, double& s, SolverShared& S, uint32_t& tot_c, double& tot_s)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    auto scan = [&](uint32_t& x, double& y) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t nc = __shfl_up_sync(0xffffffffu, x, o);
            const double ns = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) { x += nc; y = ns + y; }
        }
    };
    uint32_t ic = c;
    double is = s;
    scan(ic, is);
    const uint32_t pc = __shfl_up_sync(0xffffffffu, ic, 1);
    const double ps = __shfl_up_sync(0xffffffffu, is, 1);
    __syncthreads();
    if (lane == 31) { S.sc[warp] = ic; S.ss[warp] = is; }
    __syncthreads();
    if (warp == 0) {
        uint32_t wc = lane < nw ? S.sc[lane] : 0u;
        double ws = lane < nw ? S.ss[lane] : 0.0;
        scan(wc, ws);
        __syncwarp();
        S.sc[lane] = wc;
        S.ss[lane] = ws;
    }
    __syncthreads();
    tot_c = S.sc[31];
    tot_s = S.ss[31];
    const uint32_t bc = warp > 0 ? S.sc[warp - 1] : 0u;
    const double bs = warp > 0 ? S.ss[warp - 1] : 0.0;
    c = bc + (lane > 0 ? pc : 0u);
    s = lane > 0 ? (warp > 0 ? bs + ps : ps) : bs;
}

// ---------------------------------------------------------------------------
// Order statistics of up to kSortN values in shared memory.  The values are grouped by cells, a monotone
// function of the value with about one value to a cell, in ascending order of the cells and in any order
// inside one; a rank is found by a search over the cells and a selection inside its cell, both by a warp.
// (Nothing is sorted: a level needs one rank, and the sums before it need only know which values are
// smaller.)
// ---------------------------------------------------------------------------
struct CellIndex {
    float* sv;      // the values, at padded positions
    uint32_t* end;  // [nc] position after the last value of every cell; nc = 1024, 2048 ... 8192
    double* pre;    // [i] sum of the first i << chunk values
    int n, nc, chunk;
};

// Position i of the values: two words of padding after every sixteen, so that threads that read runs of eight or sixteen
// values side by side meet in no bank.
__device__ __forceinline__ int index_at_word(int i) { return i + ((i >> 4) << 1); }

// Shared memory: the list of the keys, later the prefix sums in its place; cells; values.
constexpr int kIndexCells = 8192;
constexpr size_t kOffIndexEnd = (size_t)kSortN * 4 + 16;
constexpr size_t kOffIndexValues = kOffIndexEnd + (size_t)kIndexCells * 4;
constexpr size_t kIndexBytes = kOffIndexValues + ((size_t)kSortN / 16 * 18) * 4;

__device__ __forceinline__ CellIndex index_at(int n)
{
    CellIndex X;
    X.pre = reinterpret_cast<double*>(smem);
    X.end = reinterpret_cast<uint32_t*>(smem + kOffIndexEnd);
    X.sv = reinterpret_cast<float*>(smem + kOffIndexValues);
    X.n = n;
    // two cells or more per value, as far as there are that many (a power of two from 1024 on): clearing and adding up more cells
    // takes longer than selecting in fuller ones saves (ResNet-50 bucket 147.6 us with 16,384, 146.2 with 8192 and with 4096)
    X.nc = min(max(1 << (32 - __clz(2 * n - 1)), 1024), kIndexCells);
    X.chunk = max(32 - __clz((n - 1) / (int)blockDim.x), 1);
    return X;
}

// cells(i, c, v): cells and values of the four values i[0..3] of n, which may lie where the prefix sums go.  Called by every
// thread of the CTA.
//   What bounds it: the latency of its six barriers and of instructions run once.  So four values of a thread are
// in flight at a time, the cells are added up without a loop, and only the positions that there are are summed (a fixed
// 16,384 positions took 2.3 us of the 13 us for 300 values).
constexpr int kIndexCols = 4;  // values of a thread in flight

template <class Cells>
__device__ __forceinline__ void index_build(const CellIndex& X, SolverShared& S, Cells cells)
{
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    uint4* rows = reinterpret_cast<uint4*>(X.end);
    for (int i = tid; i < X.nc / 4; i += nt) rows[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    constexpr int kCols = kIndexCols;
    auto four = [&](int i0, uint32_t (&c)[kCols], float (&v)[kCols]) {
        int i[kCols];
#pragma unroll
        for (int u = 0; u < kCols; ++u) i[u] = min(i0 + u * nt, X.n - 1);
        cells(i, c, v);
    };
#pragma unroll 1
    for (int i0 = tid; i0 < X.n; i0 += kCols * nt) {
        uint32_t c[kCols];
        float v[kCols];
        four(i0, c, v);
#pragma unroll
        for (int u = 0; u < kCols; ++u)
            if (i0 + u * nt < X.n) atomicAdd(X.end + c[u], 1u);
    }
    __syncthreads();
    {
        // exclusive sums over the cells, in place: a warp takes consecutive rows of 128 cells, kRows at a time
        constexpr int kRows = 4;
        const int nrows = X.nc >> 7, per = (nrows + nw - 1) / nw;
        const int r0 = min(warp * per, nrows), r1 = min(r0 + per, nrows);
        uint32_t mine = 0u;
#pragma unroll 1
        for (int q = r0; q < r1; ++q) {
            const uint4 w = rows[q * 32 + lane];
            mine += (w.x + w.y) + (w.z + w.w);
        }
        mine = __reduce_add_sync(0xffffffffu, mine);
        if (lane == 0) S.below[warp] = mine;
        __syncthreads();
        uint32_t run = __reduce_add_sync(0xffffffffu, lane < warp ? S.below[lane] : 0u);
#pragma unroll 1
        for (int q = r0; q < r1; q += kRows) {
            uint4 w[kRows];
            uint32_t own[kRows], inc[kRows];
#pragma unroll
            for (int u = 0; u < kRows; ++u) {
                w[u] = q + u < r1 ? rows[(q + u) * 32 + lane] : make_uint4(0u, 0u, 0u, 0u);
                own[u] = inc[u] = (w[u].x + w[u].y) + (w[u].z + w[u].w);
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
                for (int u = 0; u < kRows; ++u) {
                    const uint32_t nb = __shfl_up_sync(0xffffffffu, inc[u], o);
                    if (lane >= o) inc[u] += nb;
                }
            }
#pragma unroll
            for (int u = 0; u < kRows; ++u) {
                uint4 x;
                x.x = run + inc[u] - own[u]; x.y = x.x + w[u].x; x.z = x.y + w[u].y; x.w = x.z + w[u].z;
                run += __shfl_sync(0xffffffffu, inc[u], 31);
                if (q + u < r1) rows[(q + u) * 32 + lane] = x;
            }
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int i0 = tid; i0 < X.n; i0 += kCols * nt) {
        uint32_t c[kCols], at[kCols];
        float v[kCols];
        four(i0, c, v);
#pragma unroll
        for (int u = 0; u < kCols; ++u)
            if (i0 + u * nt < X.n) at[u] = atomicAdd(X.end + c[u], 1u);
#pragma unroll
        for (int u = 0; u < kCols; ++u)
            if (i0 + u * nt < X.n) X.sv[index_at_word((int)at[u])] = v[u];
    }
    __syncthreads();
    // fp64 sums before every run of 2^chunk positions, one run a thread
    const int p0 = tid << X.chunk;
    double ls = 0.0;
    if (p0 < X.n) {
#pragma unroll 1
        for (int i = p0; i < min(p0 + (1 << X.chunk), X.n); i += 2) {
            const float2 w = *reinterpret_cast<const float2*>(X.sv + index_at_word(i));
            ls += (double)w.x;
            if (i + 1 < X.n) ls += (double)w.y;
        }
    }
    const int used = (X.n + (32 << X.chunk) - 1) >> (5 + X.chunk);  // warps that have any
    if (warp < used) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double nb = __shfl_up_sync(0xffffffffu, ls, o);
            if (lane >= o) ls = nb + ls;
        }
        if (lane == 31) S.ss[warp] = ls;
    }
    __syncthreads();
    if (warp < used) {
        const double up = __shfl_up_sync(0xffffffffu, ls, 1);
        const double before = warp > 0 ? warp_sum(lane < warp ? S.ss[lane] : 0.0) : 0.0;
        X.pre[tid] = lane > 0 ? before + up : before;
        if (lane == 31 && warp == used - 1) X.pre[tid + 1] = before + ls;
    }
    __syncthreads();
}

constexpr size_t kSolveBytes = kIndexBytes + sizeof(SolverShared);
static_assert(kIndexBytes % 16 == 0 && sizeof(SolverShared) % 16 == 0, "structures in the dynamic shared memory are aligned");
__device__ __forceinline__ SolverShared& sel_state() { return *reinterpret_cast<SolverShared*>(smem + kIndexBytes); }

// floor(T), T = sum_{L <= v <= R} (v - L) / (R - L) from the prefix sums s_r and s_l at the ends of a segment of nseg values.  Where T is
// an integer (always one where nothing lies between L and R), the rounding of the sums may put it a little below:
// what is within their rounding of the next integer counts as that.
__device__ __forceinline__ double floor_of_t(double s_r, double s_l, double lval, double width, double nseg)
{
    const double low = lval * nseg, a = (s_r - s_l) - low, k = floor(a / width);
    return (k + 1.0) * width - a <= 0x1p-49 * (fabs(s_r) + fabs(s_l) + fabs(low)) ? k + 1.0 : k;
}

struct Ranked {
    float v;
    int i_lt, i_le;    // #{values < v}, #{values <= v}
    double s_lt, s_le; // their sums
};

// Sum of the values before position a <= n, by the 32 lanes of a warp.
__device__ __forceinline__ double index_before(const CellIndex& X, int a)
{
    const int lane = threadIdx.x & 31, q = a >> X.chunk, first = q << X.chunk;
    double x = first + lane < a ? (double)X.sv[index_at_word(first + lane)] : 0.0;
    for (int o = (1 << X.chunk) >> 1; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return __shfl_sync(0xffffffffu, x, 0) + X.pre[q];
}

// The value of ascending rank p, by the 32 lanes of a warp.
__device__ __forceinline__ Ranked index_select(const CellIndex& X, int p)
{
    const int lane = threadIdx.x & 31;
    // the cell that holds rank p: 32 probes in each of three steps (the first ones shifted so that they lie in different banks)
    const int s1 = X.nc >> 5, s2 = X.nc >> 10;
    const int k1 = __popc(__ballot_sync(0xffffffffu, (int)X.end[(lane + 1) * s1 - 1 - lane] <= p));
    int c = k1 > 0 ? k1 * s1 - k1 + 1 : 0;
    const int i2 = c + (lane + 1) * s2 - 1;
    c += s2 * __popc(__ballot_sync(0xffffffffu, i2 < X.nc && (int)X.end[min(i2, X.nc - 1)] <= p));
    if (s2 > 1) c += __popc(__ballot_sync(0xffffffffu, lane < s2 && (int)X.end[min(c + lane, X.nc - 1)] <= p));
    const int a = c > 0 ? (int)X.end[c - 1] : 0, b = (int)X.end[c], k = p - a;
    Ranked r;
    int lt = 0, eq = 0;
    const double before = index_before(X, a);
    double s = 0.0;
    if (b - a <= 32) {
        const float v = a + lane < b ? X.sv[index_at_word(a + lane)] : __int_as_float(0x7f800000);
#pragma unroll 1
        for (int j = 0; j < b - a; ++j) {
            const float w = __shfl_sync(0xffffffffu, v, j);
            if (w < v) {
                ++lt;
                s += (double)w;
            }
            eq += w == v ? 1 : 0;
        }
        const int src = (__ffs(__ballot_sync(0xffffffffu, a + lane < b && lt <= k && k < lt + eq)) - 1) & 31;
        r.v = __shfl_sync(0xffffffffu, v, src);
        lt = __shfl_sync(0xffffffffu, lt, src);
        eq = __shfl_sync(0xffffffffu, eq, src);
        s = __shfl_sync(0xffffffffu, s, src);
    } else {
        // a crowded cell (mostly one value many times over): its keys are bisected bit by bit
        uint32_t key = 0u;
#pragma unroll 1
        for (int bit = 31; bit >= -1; --bit) {
            const uint32_t cand = bit >= 0 ? key | (1u << bit) : key;
            int n_lt = 0, n_eq = 0;
#pragma unroll 1
            for (int i = a + lane; i < b; i += 32) {
                const float w = X.sv[index_at_word(i)];
                const uint32_t wk = float_to_key(w);
                n_lt += wk < cand ? 1 : 0;
                if (bit < 0) {
                    n_eq += wk == cand ? 1 : 0;
                    if (wk < cand) s += (double)w;
                }
            }
            n_lt = (int)__reduce_add_sync(0xffffffffu, (uint32_t)n_lt);
            if (bit >= 0) {
                if (n_lt <= k) key = cand;
            } else {
                lt = n_lt;
                eq = (int)__reduce_add_sync(0xffffffffu, (uint32_t)n_eq);
            }
        }
        r.v = key_to_float(key);
        s = warp_sum(s);
    }
    r.i_lt = a + lt;
    r.i_le = a + lt + eq;
    r.s_lt = before + s;
    r.s_le = r.s_lt + (double)r.v * (double)eq;
    return r;
}

// Levels from the indexed values: those of m intervals, which begin at positions S.start with sum S.pre before them and have
// S.before elements of the whole tensor (n of them, sum stot) below them, sum iv[].sbefore.  ORQ: the open levels of
// S.lv, one warp per level, one depth of Algorithm 1 at a time.  BinGrad-pb: the sign change of g.
// Called by every thread of the CTA.
__device__ __noinline__ void levels_from_index(int values, int m, bool pb, int s,
                                               double n, double stot, int t, float* __restrict__ levels,
                                               int32_t* __restrict__ status)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    SolverShared& S = sel_state();
    const Interval* iv = S.niv;
    const CellIndex X = index_at(values);  // (made again: a reference would put it into local memory)
    if (!pb) {
        static_assert(kSelWarps >= kMaxLv - 1, "one warp per interior level");
        const int q = warp;
#pragma unroll 1
        for (int stride = (s - 1) >> 1; stride >= 1; stride >>= 1) {
            if (q < s - 1 && q >= stride && ((q - stride) & (2 * stride - 1)) == 0 && !S.lv[q].exact) {
                const LvInfo &L = S.lv[q - stride], &R = S.lv[q + stride];
                LvInfo& o = S.lv[q];
                const double lval = L.val, width = R.val - lval;
                const uint32_t le = (uint32_t)R.c_le, lt = (uint32_t)L.c_lt;
                if (!(width > 0.0)) {
                    if (lane == 0) o = L;
                } else {
                    const double nseg = (double)(le - lt);
                    const uint32_t k = (uint32_t)fmin(fmax(floor_of_t(R.s_le, L.s_lt, lval, width, nseg), 0.0), nseg - 1.0), p = le - 1u - k;
                    // the interval that holds rank p: the last one that begins at or before it
                    int j = __popc(__ballot_sync(0xffffffffu, S.before[lane] <= p)) - 1;
                    if (m > 32) j += __popc(__ballot_sync(0xffffffffu, S.before[lane + 32] <= p));
                    const int i = j >= 0 ? S.start[j] + (int)(p - S.before[j]) : -1;
                    if (i < 0 || i >= S.start[j + 1]) {
                        if (lane == 0) { o = L; S.internal = 1; }
                    } else {
                        const Ranked r = index_select(X, i);
                        if (lane == 0) {
                            const uint32_t cb = S.before[j] - (uint32_t)S.start[j];
                            const double sb = iv[j].sbefore, pre = S.pre[j];
                            o.val = (double)r.v;
                            o.c_lt = cb + (uint32_t)r.i_lt;
                            o.c_le = cb + (uint32_t)r.i_le;
                            o.s_lt = sb + (r.s_lt - pre);
                            o.s_le = sb + (r.s_le - pre);
                        }
                    }
                }
            }
            __syncthreads();
        }
        const bool fail = S.internal != 0;
        if ((int)threadIdx.x < s) levels[(int64_t)t * s + threadIdx.x] = fail ? 0.f : (float)S.lv[threadIdx.x].val;
        if (threadIdx.x == 0 && fail) status[t] |= OGQ_ST_INTERNAL;
        return;
    }
    // BinGrad-pb: the values with g(x) = x n - sum_{|v| >= x} |v| <= 0 come first.  Two ranks that enclose the last of them, from the
    // first value w of every run of positions: what lies below w's cell has at least the sum of the whole runs before
    // that cell, what lies below w at most that of the runs up to the cell's end.  Then a warp per candidate rank.
    // (The ranks by rounds of 32 candidates alone took 16,000 cycles for 16,384 values: three rounds and a last selection.)
    const int nw = blockDim.x >> 5;
    int lo = -1, hi = X.n;  // g <= 0 at lo (or lo = -1), g > 0 at hi (or hi = n)
    {
        const int i = (int)threadIdx.x << X.chunk;
        if (i < X.n) {
            const double w = (double)X.sv[index_at_word(i)];
            int c = 0;  // w's cell: the first that ends after i
#pragma unroll 1
            for (int step = X.nc >> 1; step >= 1; step >>= 1)
                if ((int)X.end[c + step - 1] <= i) c += step;
            const int a = c > 0 ? (int)X.end[c - 1] : 0, b = (int)X.end[c], j = c / (X.nc / m);
            const double shift = stot - (iv[j].sbefore - S.pre[j]), x = w * n, eps = 1e-11 * (x + stot);
            if (x - (shift - X.pre[(b + (1 << X.chunk) - 1) >> X.chunk]) < -eps) lo = a;
            if (x - (shift - X.pre[a >> X.chunk]) > eps) hi = b - 1;
        }
        lo = __reduce_max_sync(0xffffffffu, lo);
        hi = __reduce_min_sync(0xffffffffu, hi);
        if (lane == 0) { S.sc[warp] = (uint32_t)lo; S.below[warp] = (uint32_t)hi; }
        __syncthreads();
        lo = __reduce_max_sync(0xffffffffu, lane < nw ? (int)S.sc[lane] : -1);
        hi = __reduce_min_sync(0xffffffffu, lane < nw ? (int)S.below[lane] : X.n);
        __syncthreads();
    }
    double b1 = 0.0;
#pragma unroll 1
    while (true) {
        const bool last = hi - lo <= nw;
        const int step = last ? 1 : (hi - lo + nw - 1) / nw, i = (last ? lo : lo + 1) + warp * step;
        bool below = i < 0;
        if (below) {
            b1 = fp64_div(stot - iv[0].sbefore, n);  // the zero when it lies below every value of the bracket
        } else if (i < hi) {
            const Ranked r = index_select(X, i);
            const int j = __popc(__ballot_sync(0xffffffffu, lane < m && S.start[lane] <= i)) +
                          __popc(__ballot_sync(0xffffffffu, lane + 32 < m && S.start[lane + 32] <= i)) - 1;
            const double x = (double)r.v, before = iv[j].sbefore + (r.s_lt - S.pre[j]);
            below = x * n - (stot - before) <= 0.0 || (last && warp == 0);  // (at lo, known)
            if (last) {
                const double up = fp64_div(stot - (iv[j].sbefore + (r.s_le - S.pre[j])), n);
                b1 = up > x ? up : x;
            }
        }
        if (lane == 0) { S.below[warp] = below ? 1u : 0u; S.ss[warp] = b1; }
        __syncthreads();
        const int k = __popc(__ballot_sync(0xffffffffu, lane < nw && S.below[lane]));
        if (last) {
            b1 = S.ss[k - 1];
            break;
        }
        __syncthreads();
        const int nhi = lo + 1 + k * step;
        if (k > 0) lo += 1 + (k - 1) * step;
        if (nhi < hi) hi = nhi;
    }
    if (threadIdx.x == 0) {
        if (S.internal) { status[t] |= OGQ_ST_INTERNAL; b1 = 0.0; }
        levels[2 * t] = -(float)b1;
        levels[2 * t + 1] = (float)b1;
    }
}

// Finishes the tensor from the keys inside the intervals S.niv, which fit kSortN: src[0 .. src_cnt) are these keys as a copy-only pass
// wrote them (packed; src is 16-byte aligned and readable to the end of its last 16 bytes), or keys among which they are.
__device__ __noinline__ void finish_from_keys(TState* st, int t, bool pb, int s, const uint32_t* src, int src_cnt, bool packed,
                                              float* __restrict__ levels, int32_t* __restrict__ status)
{
    const int tid = threadIdx.x, lane = tid & 31, nt = blockDim.x;
    SolverShared& S = sel_state();
    uint32_t* list = reinterpret_cast<uint32_t*>(smem);
    __syncthreads();  // S.nm and S.niv are complete; the shared memory is free
    const int m = S.nm;
    int c = src_cnt;
    if (packed) {
        const uint32_t to = (uint32_t)__cvta_generic_to_shared(list);
#pragma unroll 1
        for (int i = tid; i < (src_cnt + 3) / 4; i += nt)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(to + 16u * (uint32_t)i), "l"(src + 4 * (size_t)i) : "memory");
    }
    if (tid < kMaxIv) {
        const bool real = tid < m;
        S.place[tid].x = real ? S.niv[tid].klo : 0xffffffffu;  // (no key has this value: NaN)
        S.place[tid].y = real ? S.niv[tid].khi : 0u;
        S.before[tid] = real ? (uint32_t)S.niv[tid].cbefore : 0xffffffffu;
    }
    if (tid == 0) { S.n_keys = 0; S.internal = 0; }
    if (packed) asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    constexpr int kCols = kIndexCols;
    if (!packed) {
        int top = 1;
        while (top < m) top <<= 1;
#pragma unroll 1
        for (int i0 = tid & ~31; i0 < src_cnt; i0 += kCols * nt) {
            uint32_t k[kCols];
#pragma unroll
            for (int u = 0; u < kCols; ++u) {
                const int i = i0 + u * nt + lane;
                k[u] = i < src_cnt ? __ldcg(src + i) : 0u;
            }
            int j[kCols];
#pragma unroll
            for (int u = 0; u < kCols; ++u) j[u] = 0;
#pragma unroll 1
            for (int step = top >> 1; step >= 1; step >>= 1) {
#pragma unroll
                for (int u = 0; u < kCols; ++u)
                    if (S.place[j[u] + step].x <= k[u]) j[u] += step;
            }
#pragma unroll
            for (int u = 0; u < kCols; ++u) {
                const uint4 at = S.place[j[u]];
                const bool in = i0 + u * nt + lane < src_cnt && k[u] >= at.x && k[u] <= at.y;
                const unsigned b = __ballot_sync(0xffffffffu, in);
                if (b) {
                    int pos = 0;
                    if (lane == 0) pos = atomicAdd(&S.n_keys, __popc(b));
                    pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(b & ((1u << lane) - 1u));
                    if (in && pos < kSortN) list[pos] = (uint32_t)j[u] << kRelBits | ((k[u] - at.x) & ((1u << kRelBits) - 1u));
                }
            }
        }
        __syncthreads();
        c = S.n_keys;
        if (c > kSortN) { c = kSortN; if (tid == 0) S.internal = 1; }
    }
    const CellIndex X = index_at(c);
    if (tid < m) {
        // equal shares of the cells: an interval is a narrow slice of a binade, its values are spread evenly
        const uint32_t share = (uint32_t)(X.nc / m);
        S.place[tid].z = tid * share;
        S.place[tid].w = (uint32_t)max(0, 32 - __clz((S.place[tid].y - S.place[tid].x) / share));
    }
    // (index_build has a barrier before the first cell is asked for)
    index_build(X, S, [&](const int (&i)[kCols], uint32_t (&cell)[kCols], float (&v)[kCols]) {
        uint32_t k[kCols];
#pragma unroll
        for (int u = 0; u < kCols; ++u) k[u] = list[i[u]];
#pragma unroll
        for (int u = 0; u < kCols; ++u) {
            const uint4 at = S.place[k[u] >> kRelBits];
            const uint32_t rel = k[u] & ((1u << kRelBits) - 1u);
            cell[u] = at.z + (rel >> at.w);
            v[u] = sel_key_to_float(at.x + rel);
        }
    });
    for (int j = tid >> 5; j <= m; j += nt >> 5) {
        // where interval j begins: after the last value of the cell before its first
        const int a = j == m ? c : (j > 0 ? (int)X.end[S.place[j].z - 1u] : 0);
        const double x = index_before(X, a);
        if (lane == 0) {
            S.start[j] = a;
            if (j < m) S.pre[j] = x;
        }
    }
    __syncthreads();
    levels_from_index(c, m, pb, s, (double)S.view.n, S.view.stot, t, levels, status);
    if (tid == 0) st->done = 1;
}

// Small tensors: all values indexed, the definitions applied directly.
__device__ void small_tensor(const float* __restrict__ src, int n, int t, bool pb, int s, float* __restrict__ levels,
                             int32_t* __restrict__ status, float tau)
{
    SolverShared& S = sel_state();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x, nw = nt >> 5;
    float* values = reinterpret_cast<float*>(smem);  // clipped, -0 as 0, magnitudes for BinGrad-pb
    uint32_t kmin = 0xffffffffu, kmax = 0u, sum = 0u;
    constexpr int kCols = kIndexCols;
    // (asynchronous copies: one latency of DRAM for all of a thread's values; four at a time in registers, 16,384 values took
    // 17,000 cycles to load)
    const uint32_t to = (uint32_t)__cvta_generic_to_shared(values);
    const int whole = ((uintptr_t)src & 15) == 0 ? n & ~3 : 0;
#pragma unroll 1
    for (int i = 4 * tid; i < whole; i += 4 * nt)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(to + 4u * (uint32_t)i), "l"(src + i) : "memory");
#pragma unroll 1
    for (int i = whole + tid; i < n; i += nt)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" :: "r"(to + 4u * (uint32_t)i), "l"(src + i) : "memory");
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
#pragma unroll 4
    for (int i = tid; i < n; i += nt) {
        const float x = values[i];
        float v = copysignf(fminf(fabsf(x), tau), x) + 0.0f;
        if (pb) v = fabsf(v);
        values[i] = v;
        const uint32_t k = float_to_key(v);
        kmin = min(kmin, k);
        kmax = max(kmax, k);
        sum += (__float_as_uint(v) & 0x7fffffffu) >> 16;
    }
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0) S.place[warp] = make_uint4(kmin, kmax, sum, 0u);
    __syncthreads();
    const uint4 w = S.place[lane & (nw - 1)];
    kmin = __reduce_min_sync(0xffffffffu, w.x);
    kmax = __reduce_max_sync(0xffffffffu, w.y);
    sum = __reduce_add_sync(0xffffffffu, lane < nw ? w.z : 0u);
    const float vmin = key_to_float(kmin), vmax = key_to_float(kmax);
    const int nl = pb ? 2 : s;
    // (keys order Inf and NaN beyond the finite values at either end)
    const bool bad = kmax >= 0xff800000u || kmin <= 0x007fffffu;
    if (bad || kmin == kmax) {
        // non-finite, or all values equal: level = value (BinGrad-pb: b_1 = the magnitude, b_0 = b_1 = 0 for zeros)
        if (tid < nl) levels[(int64_t)t * nl + tid] = bad ? 0.f : pb ? (tid == 0 ? -vmax : vmax) : vmax;
        if (tid == 0) status[t] = bad ? OGQ_ST_NONFINITE : (!pb || vmax == 0.f) ? OGQ_ST_CONSTANT : 0;
        return;
    }
    const CellIndex X = index_at(n);
    const MagnitudeCells cell((uint32_t)((float)sum / (float)n), fmaxf(fabsf(vmin), fabsf(vmax)), !pb, (uint32_t)X.nc);
    index_build(X, S, [&](const int (&i)[kCols], uint32_t (&c)[kCols], float (&v)[kCols]) {
#pragma unroll
        for (int u = 0; u < kCols; ++u) {
            v[u] = values[i[u]];
            c[u] = cell(v[u]);
        }
    });
    // (the total the way index_select adds prefixes up)
    const double stot = index_before(X, n);
    if (tid < kMaxIv) S.before[tid] = tid == 0 ? 0u : 0xffffffffu;
    if (tid == 0) {
        S.internal = 0;
        S.start[0] = 0; S.start[1] = n; S.pre[0] = 0.0;
        S.niv[0].sbefore = 0.0;
        status[t] = 0;
    }
    if (tid < s) {
        LvInfo& l = S.lv[tid];
        l.exact = tid == 0 || tid == s - 1;
        l.val = (double)(tid == 0 ? vmin : vmax);
        l.key = tid == 0 ? kmin : kmax;
        l.c_lt = 0; l.s_lt = 0.0;
        l.c_le = n; l.s_le = stot;
    }
    __syncthreads();
    levels_from_index(n, 1, pb, s, (double)n, stot, t, levels, status);
}

// What the finish of a tensor needs from its state, for a tensor whose last pass only copied the keys inside its intervals
// (TState::compact_only).  Called by every thread of the CTA; every load is issued before the first is waited for.
// Intervals beyond st->m are not used.
__device__ __forceinline__ void finish_load(const TState* st, bool pb, int s, SolverShared& S)
{
    const int tid = threadIdx.x;
    if (tid < kMaxIv) S.niv[tid] = st->iv[tid];
    if (!pb && tid >= 64 && tid - 64 < s) {
        const ExactLv& e = st->lv[tid - 64];
        LvInfo& l = S.lv[tid - 64];
        l.exact = e.exact; l.key = e.key; l.val = (double)sel_key_to_float(e.key);
        l.c_lt = e.c_lt; l.c_le = e.c_le; l.s_lt = e.s_lt; l.s_le = e.s_le;
    }
    if (tid == 96) {
        S.view.n = st->n;
        S.view.stot = st->stot;
        S.nm = st->m;
    }
}

// Finishes such a tensor.
__device__ void finish_sorted(TState* st, int t, bool pb, int s, const uint32_t* copied, float* __restrict__ levels,
                              int32_t* __restrict__ status, int cursor_idx)
{
    const long long cand = __ldcg(&st->cand), src_cnt = (long long)__ldcg(&st->cursor[cursor_idx]);
    __syncthreads();
    finish_load(st, pb, s, sel_state());
    finish_from_keys(st, t, pb, s, copied, (int)min(src_cnt, cand), true, levels, status);
}

// Shared memory of a solver pass: the prefix arrays over the slots, and the raw cells as they come from L2.
constexpr size_t kOffSpre = (kSlots * sizeof(uint32_t) + 15) / 16 * 16;
constexpr size_t kOffSlotIv = kOffSpre + kSlots * sizeof(double);
constexpr size_t kOffRawSum = (kOffSlotIv + kSlots + 15) / 16 * 16;
constexpr size_t kOffRawCnt = kOffRawSum + kCells * sizeof(unsigned long long);
constexpr size_t kPrefixBytes = kOffRawCnt + kCells * sizeof(uint32_t);
static_assert(kPrefixBytes <= kIndexBytes && kOffStage + 2 * kSmemStage <= kIndexBytes, "the index takes the most shared memory");

// Prefix arrays over all slots of the intervals S.iv (S.view.m of them): counts and sums of the elements
// before every slot.  A thread takes consecutive slots; a slot's cell is its index minus the number of
// intervals before it (every interval has one end slot).
__device__ __forceinline__ void solver_prefix(SolverShared& S, const uint32_t* gcnt, const unsigned long long* glsum, bool first)
{
    uint32_t* cpre = reinterpret_cast<uint32_t*>(smem);
    double* spre = reinterpret_cast<double*>(smem + kOffSpre);
    uint8_t* slot_iv = smem + kOffSlotIv;
    unsigned long long* raw_sum = reinterpret_cast<unsigned long long*>(smem + kOffRawSum);
    uint32_t* raw_cnt = reinterpret_cast<uint32_t*>(smem + kOffRawCnt);
    const int tid = threadIdx.x, nt = blockDim.x, m = S.view.m;
    const int ncells = S.iv[m - 1].cellbase + S.iv[m - 1].ncell, nslots = ncells + m;
    {
        constexpr int kC = (kCells / 4 + kSelThreads - 1) / kSelThreads, kL = (kCells / 2 + kSelThreads - 1) / kSelThreads;
        uint4 c[kC];
        ulonglong2 l[kL];
#pragma unroll
        for (int u = 0; u < kC; ++u)
            if ((tid + u * nt) * 4 < ncells) c[u] = __ldcg(reinterpret_cast<const uint4*>(gcnt) + tid + u * nt);
#pragma unroll
        for (int u = 0; u < kL; ++u)
            if ((tid + u * nt) * 2 < ncells) l[u] = __ldcg(reinterpret_cast<const ulonglong2*>(glsum) + tid + u * nt);
        if (tid < m) S.view.slotbase[tid] = S.iv[tid].cellbase + tid;
        if (tid == 0) { S.view.slotbase[m] = nslots; S.view.nslots = nslots; }
#pragma unroll
        for (int u = 0; u < kC; ++u)
            if ((tid + u * nt) * 4 < ncells) reinterpret_cast<uint4*>(raw_cnt)[tid + u * nt] = c[u];
#pragma unroll
        for (int u = 0; u < kL; ++u)
            if ((tid + u * nt) * 2 < ncells) reinterpret_cast<ulonglong2*>(raw_sum)[tid + u * nt] = l[u];
    }
    __syncthreads();
    const int per = (nslots + nt - 1) / nt;
    const int s0 = tid * per < nslots ? tid * per : nslots, s1 = s0 + per < nslots ? s0 + per : nslots;
    int j = 0;
    {
        int hi = m;
#pragma unroll 1
        while (hi - j > 1) { const int mid = (j + hi) >> 1; if (S.view.slotbase[mid] <= s0) j = mid; else hi = mid; }
    }
    uint32_t lc = 0;
    double ls = 0.0;
#pragma unroll 1
    for (int slot = s0; slot < s1; ++slot) {
        while (slot >= S.view.slotbase[j + 1]) ++j;
        slot_iv[slot] = (uint8_t)j;
        const uint32_t n = slot + 1 < S.view.slotbase[j + 1] ? raw_cnt[slot - j] : 0u;
        double x = 0.0;
        if (n) x = sel_cell_sum(S.iv[j].klo + ((uint32_t)(slot - S.view.slotbase[j]) << S.iv[j].sh), S.iv[j].sh, n, raw_sum[slot - j]);
        cpre[slot] = n;
        spre[slot] = x;
        lc += n;
        ls += x;
    }
    uint32_t tc;
    double ts;
    block_excl_scan(lc, ls, S, tc, ts);
#pragma unroll 1
    for (int slot = s0; slot < s1; ++slot) {
        const uint32_t n = cpre[slot];
        const double x = spre[slot];
        cpre[slot] = lc;
        spre[slot] = ls;
        lc += n;
        ls += x;
    }
    __syncthreads();
    if (first) return;
    // rounds >= 2: shift every interval so that it starts from the exact (count, sum) before it
    if (tid < m) {
        const int sb = S.view.slotbase[tid];
        S.offc[tid] = (uint32_t)((unsigned long long)S.iv[tid].cbefore - cpre[sb]);
        S.offs[tid] = S.iv[tid].sbefore - spre[sb];
    }
    __syncthreads();
#pragma unroll 1
    for (int slot = s0; slot < s1; ++slot) {
        cpre[slot] += S.offc[slot_iv[slot]];
        spre[slot] += S.offs[slot_iv[slot]];
    }
    __syncthreads();
}

// Q*(L, R) on the current cells, by the 32 lanes of a warp: exact when both brackets are exact and the target
// rank sits in a single-key cell, otherwise a conservative range of cells [sa, sb].  The lower half of the
// lanes works out the range's first rank and its cell, the upper half the last; both are the same when the
// brackets are exact.  Returns false on an internal inconsistency.
//   With M the elements strictly between L's cells and R's cells (count cntM, sum sumM), T = [t_L + (sumM -
// L cntM) + t_R] / (R - L), t_L and t_R the contributions of the elements of L's and R's own cells.
// (sumM - L cntM) / (R - L) decreases in L and in R, so its extremes are taken at matching corners, which
// stays tight even when a bracket is only known to lie somewhere in a sparse stretch of cells.
__device__ __noinline__ bool warp_orq_solve(int q, int stride)
{
    SolverShared& S = sel_state();
    const SolverView& v = S.view;
    const LvInfo &L = S.lv[q - stride], &R = S.lv[q + stride];
    LvInfo& out = S.lv[q];
    const int lane = threadIdx.x & 31;
    const bool upper = lane >= 16;
    if (L.exact && R.exact && !(R.val > L.val)) {
        if (lane == 0) out = L;
        return true;
    }
    const bool exact = L.exact && R.exact;
    // (an exact level's range is its value: vlo = vhi = val, and c_lt .. c_le, s_lt .. s_le its elements; one
    // that is only known as a range has the counts and sums of the whole range there)
    const long long floor_pos = L.c_lt, ceil_pos = R.c_le - 1;
    long long pos;
    if (exact) {
        const long long nseg = R.c_le - L.c_lt;
        long long k = (long long)floor_of_t(R.s_le, L.s_lt, L.val, R.val - L.val, (double)nseg);
        if (k < 0) k = 0;
        if (k > nseg - 1) k = nseg - 1;
        pos = R.c_le - 1 - k;
    } else {
        const long long Cs = L.exact ? L.c_lt : L.c_le, Ce = R.exact ? R.c_le : R.c_lt;
        const double Ss = L.exact ? L.s_lt : L.s_le, Se = R.exact ? R.s_le : R.s_lt;
        const double cntL = L.exact ? 0.0 : (double)(L.c_le - L.c_lt), cntR = R.exact ? 0.0 : (double)(R.c_le - R.c_lt);
        const double cntM = (double)(Ce - Cs), sumM = Se - Ss;
        pos = upper ? ceil_pos : floor_pos;
        if (cntM >= 0.0 && R.vlo > L.vhi) {
            double num = fmax(sumM - (upper ? L.vhi : L.vlo) * cntM, 0.0);
            num = upper ? cntR * (R.vhi - R.vlo) - num : -(cntL * (L.vhi - L.vlo) + num);
            const double den = upper ? R.vhi - L.vhi : R.vlo - L.vlo;
            const double delta = 2.0 + 1e-9 * (double)v.n;
            const double p = ceil((double)Ce + fp64_div(num, den) + (upper ? delta : -delta)) - 1.0;
            if (upper ? p < (double)pos : p > (double)pos) pos = (long long)p;
        }
        if (pos < floor_pos) pos = floor_pos;
        if (pos > ceil_pos) pos = ceil_pos;
        const long long other = __shfl_xor_sync(0xffffffffu, pos, 16);
        if (!upper && pos > other) pos = other;
        if (pos < 0) pos = 0;
        if (pos > v.n - 1) pos = v.n - 1;
    }
    // the cells of the two ranks: each half of the warp searches for the first slot whose prefix exceeds its own
    int lo = 0, hi = v.nslots;
#pragma unroll 1
    while (__any_sync(0xffffffffu, lo < hi)) {
        const int step = (hi - lo + 15) >> 4;
        const int i = lo + (lane & 15) * step;
        const unsigned b = __ballot_sync(0xffffffffu, i < hi && (long long)v.cpre[i] <= pos);
        const int k = __popc(upper ? b >> 16 : b & 0xffffu);
        const int nhi = lo + k * step;
        if (k > 0) lo += (k - 1) * step + 1;
        if (nhi < hi) hi = nhi;
    }
    // lo - 1 is the cell's slot; the end slot of an interval there means that the rank lies between two
    // intervals: the first cell after the gap for the lower rank, the last one before it for the upper
    int slot = lo - 1;
    const bool gap = slot < 0 || sel_is_end_slot(v, slot);
    if (gap) slot = (upper && !exact) ? slot - 1 : slot + 1;
    bool ok = slot >= 0 && slot < v.nslots && !(exact && gap);
    const int sa = __shfl_sync(0xffffffffu, slot, 0), sb = __shfl_sync(0xffffffffu, slot, 16);
    ok = __all_sync(0xffffffffu, ok) && sa <= sb;
    if (!ok) return false;
    // value bounds: the low end of the first cell, the high end of the last
    const int sh = sel_slot_shift(v, slot);
    const double val = (double)sel_key_to_float(sel_slot_kbase(v, slot) + (upper && sh > 0 ? (1u << sh) - 1u : 0u));
    const double vhi = __shfl_sync(0xffffffffu, val, 16);
    if (lane == 0) {
        out.exact = exact && sh == 0;
        out.key = sel_slot_kbase(v, sa);
        out.val = val;
        out.vlo = val;
        out.vhi = vhi;
        out.c_lt = v.cpre[sa];
        out.s_lt = v.spre[sa];
        out.c_le = v.cpre[sb + 1];
        out.s_le = v.spre[sb + 1];
        out.sa = sa;
        out.sb = sb;
    }
    return true;
}

// Turns the candidate cells (S.marks) into the intervals of the next round (S.niv, S.nm, S.cand): a run of
// neighbouring candidate cells is an interval, and the cell budget is shared out equally among the runs,
// each taking as many halvings of its cells as its share allows (a run that is longer than its share keeps
// its cells and the others share the rest).  Returns false when there are more than kRefineMax runs or the
// shares do not work out.  Called by the 32 lanes of warp 0.
__device__ __forceinline__ bool refine_marked(SolverShared& S)
{
    const SolverView& v = S.view;
    const int lane = threadIdx.x & 31;
    constexpr int kWords = (kSlots + 31) / 32, kWpl = (kWords + 31) / 32;
    const int w0 = lane * kWpl, w1 = w0 + kWpl < kWords ? w0 + kWpl : kWords;
    // first and last cells of runs in this lane's words: counted, then written out
    int is = 0, ie = 0, m = 0;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        int ns = 0, ne = 0;
#pragma unroll 1
        for (int w = w0; w < w1; ++w) {
            const uint32_t x = S.marks[w];
            if (x == 0u) continue;
            uint32_t a = x & ~((x << 1) | (w > 0 ? S.marks[w - 1] >> 31 : 0u));
            uint32_t b = x & ~((x >> 1) | (w + 1 < kWords ? S.marks[w + 1] << 31 : 0u));
            if (pass == 0) {
                ns += __popc(a);
                ne += __popc(b);
            } else {
                for (; a; a &= a - 1) S.pa[is++] = w * 32 + __ffs(a) - 1;
                for (; b; b &= b - 1) S.pb[ie++] = w * 32 + __ffs(b) - 1;
            }
        }
        if (pass == 0) {
            is = ns;
            ie = ne;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int a = __shfl_up_sync(0xffffffffu, is, o), b = __shfl_up_sync(0xffffffffu, ie, o);
                if (lane >= o) { is += a; ie += b; }
            }
            m = __shfl_sync(0xffffffffu, is, 31);
            if (m == 0 || m > kRefineMax) return false;
            is -= ns;
            ie -= ne;
        }
    }
    __syncwarp();
    static_assert(kRefineMax == 32, "a lane per run");
    const bool have = lane < m;
    const int pa = have ? S.pa[lane] : 0, pb = have ? S.pb[lane] : 0;
    const int len = have ? pb - pa + 1 : 0, j = have ? v.slot_iv[pa] : 0;
    int sh = have ? v.iv[j].sh : 0;
    const bool large = len > kCells / m;
    const int big = __reduce_add_sync(0xffffffffu, large ? len : 0), nbig = __popc(__ballot_sync(0xffffffffu, large));
    const int share = nbig < m ? (kCells - big) / (m - nbig) : 0;
    const int r = have && len <= share ? min(31 - __clz(share / len), sh) : 0;
    const int ncell = len << r;
    sh -= r;
    const bool progress = __any_sync(0xffffffffu, r > 0), open_shift = __any_sync(0xffffffffu, sh > 0);
    int at = ncell;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, at, o);
        if (lane >= o) at += a;
    }
    if (__shfl_sync(0xffffffffu, at, 31) > kCells || (open_shift && !progress)) return false;
    if (have) {
        const Interval& o = v.iv[j];
        Interval& ni = S.niv[lane];
        ni.sh = sh;
        ni.ncell = ncell;
        ni.klo = o.klo + ((uint32_t)(pa - v.slotbase[j]) << o.sh);
        ni.khi = ni.klo + (uint32_t)((((unsigned long long)ncell) << sh) - 1ull);
        ni.cellbase = at - ncell;
        ni.pad = 0;
        ni.cbefore = v.cpre[pa];
        ni.sbefore = v.spre[pa];
        atomicAdd((unsigned long long*)&S.cand, (unsigned long long)(v.cpre[pb + 1] - v.cpre[pa]));
    }
    if (lane == 0) S.nm = m;
    __syncwarp();
    return true;
}

// Runs one solver pass for tensor t after a pass over it is complete: prefix arrays, then the levels or a
// conservative range of cells for each, then the intervals of the next pass, or the finish when the copied
// keys inside the new intervals are few enough.  Called by every thread of the CTA; returns true when the
// tensor is finished.  S.iv, S.view.m / n / stot and S.lv describe the pass that just ended.
//   round_buf: the keys copied by the pass (null: none were), cap: words of the tensor's key region.
__device__ __noinline__ bool solver_round(TState* st, int t, uint32_t* gcnt, unsigned long long* glsum, int scheme,
                             int s, float* __restrict__ levels, int32_t* __restrict__ status,
                             unsigned* nitems, int2* items, const uint32_t* round_buf, bool enqueue, int64_t cap, int round)
{
    SolverShared& S = sel_state();
    uint32_t* cpre = reinterpret_cast<uint32_t*>(smem);
    double* spre = reinterpret_cast<double*>(smem + kOffSpre);
    const bool pb = scheme == OGQ_BINGRAD_PB;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x, nt = blockDim.x;

    if (tid == 0) {
        S.view.iv = S.iv;
        S.view.slot_iv = smem + kOffSlotIv;
        S.view.cpre = cpre;
        S.view.spre = spre;
        S.done = 0; S.nm = -100; S.internal = 0; S.cand = 0; S.nopen = 0;
        S.pb_a = -1; S.pb_b = -1; S.pb_c = -1;
    }
    for (int i = tid; i < (kSlots + 31) / 32; i += nt) S.marks[i] = 0u;
    __syncthreads();
    solver_prefix(S, gcnt, glsum, round == 1);
    const int nslots = S.view.nslots;
    if (round == 1) {
        if (tid == 0) {
            const double stot = spre[nslots - 1];
            S.view.stot = stot;
            st->stot = stot;
            LvInfo& l = S.lv[pb ? 1 : s - 1];
            l.c_le = S.view.n;
            l.s_le = stot;
            if ((long long)cpre[nslots - 1] != S.view.n) S.internal = 1;
        }
        __syncthreads();
    }
    const double stot = S.view.stot;
    int range_a = -1, range_b = -1;  // this warp's open range

    if (!pb) {
        // one warp per level, one depth of Algorithm 1 at a time
        static_assert(kSelWarps >= kMaxLv - 1, "one warp per interior level");
#pragma unroll 1
        for (int stride = (s - 1) >> 1; stride >= 1; stride >>= 1) {
            const int q = warp;
            if (q < s - 1 && q >= stride && ((q - stride) & (2 * stride - 1)) == 0 && !S.lv[q].exact) {
                const bool ok = warp_orq_solve(q, stride);
                __syncwarp();
                if (!ok) {
                    if (lane == 0) S.internal = 1;
                } else if (!S.lv[q].exact) {
                    range_a = S.lv[q].sa;
                    range_b = S.lv[q].sb;
                    if (lane == 0) S.nopen = 1;
                }
            }
            __syncthreads();
        }
        if (tid < s) {
            ExactLv& e = st->lv[tid];
            const LvInfo& l = S.lv[tid];
            e.exact = l.exact; e.key = l.key; e.c_lt = l.c_lt; e.c_le = l.c_le; e.s_lt = l.s_lt; e.s_le = l.s_le;
        }
    } else if (!S.internal && stot > 0.0) {
        // bracket of the sign change of g, evaluated at the lower edge of every cell
        int a = -1, b = -1, cs = -1;
#pragma unroll 1
        for (int sl = tid; sl < nslots; sl += nt) {
            if (sel_is_end_slot(S.view, sl)) continue;
            double x;
            const double g = sel_pb_g(S.view, sl, &x);
            if (!(x < INFINITY)) continue;
            const double eps = 1e-11 * (x * (double)S.view.n + stot);
            if (g < -eps) a = sl;
            if (g <= eps) b = sl;
            if (g <= 0.0) cs = sl;
        }
        if (a >= 0) atomicMax(&S.pb_a, a);
        if (b >= 0) atomicMax(&S.pb_b, b);
        if (cs >= 0) atomicMax(&S.pb_c, cs);
        __syncthreads();
        a = S.pb_a < 0 ? 0 : S.pb_a;
        b = S.pb_b < a ? a : S.pb_b;
        cs = S.pb_c < a ? a : S.pb_c;
        if (cs > b) cs = b;
        bool coarse = false;  // some cell of the bracket holds more than one key
        for (int sl = a + tid; sl <= b; sl += nt)
            coarse |= !sel_is_end_slot(S.view, sl) && sel_slot_shift(S.view, sl) != 0;
        coarse = __syncthreads_or(coarse);
        if (cpre[b + 1] == cpre[a]) {
            // no element in the bracket: g is zero between two magnitudes
            if (tid == 0) {
                const float b1 = (float)((stot - spre[a]) / (double)S.view.n);
                levels[2 * t] = -b1; levels[2 * t + 1] = b1;
            }
        } else if (!coarse && !sel_is_end_slot(S.view, cs)) {
            if (tid == 0) {
                const float b1 = (float)sel_pb_final(S.view, cs);
                levels[2 * t] = -b1; levels[2 * t + 1] = b1;
            }
        } else {
            if (warp == 0) { range_a = a; range_b = b; }
            if (tid == 0) S.nopen = 1;
        }
        __syncthreads();
    }
    const bool fail = S.internal != 0, zero = pb && !fail && !(stot > 0.0);
    const bool capped = round + 1 > kMaxRounds && S.nopen;
    if (fail || zero || !S.nopen || capped) {
        const int nl = pb ? 2 : s;
        if (fail || zero || capped) {
            // unresolved: zeros rather than garbage
            if (tid < nl) levels[(int64_t)t * nl + tid] = 0.f;
            if (tid == 0) status[t] |= fail ? OGQ_ST_INTERNAL : zero ? OGQ_ST_CONSTANT : OGQ_ST_ITER_CAP;
        } else if (!pb && tid < s) {
            levels[(int64_t)t * s + tid] = sel_key_to_float(S.lv[tid].key);
        }
        if (tid == 0) st->done = 1;
        __threadfence();
        __syncthreads();
        return true;
    }
    // candidate cells: the populated cells of the open ranges
    if (range_a >= 0) {
#pragma unroll 1
        for (int c0 = range_a & ~31; c0 <= range_b; c0 += 32) {
            const int c = c0 + lane;
            const bool in = c >= range_a && c <= range_b && !sel_is_end_slot(S.view, c) && cpre[c + 1] != cpre[c];
            const uint32_t w = __ballot_sync(0xffffffffu, in);
            if (lane == 0 && w) atomicOr(&S.marks[c0 >> 5], w);
        }
    }
    __syncthreads();
    if (warp == 0) {
        const bool ok = refine_marked(S);
        if (lane == 0 && !ok) {
            // too many scattered cells: the general single-thread routine, which may keep empty stretches
            int nr = 0, ra[kMaxLv], rb[kMaxLv];
            if (pb) { ra[0] = range_a; rb[0] = range_b; nr = 1; }
            else
                for (int q = 1; q < s - 1; ++q)
                    if (!S.lv[q].exact) { ra[nr] = S.lv[q].sa; rb[nr] = S.lv[q].sb; ++nr; }
            S.nm = sel_refine(S.view, nr, ra, rb, !pb, S.niv, &S.cand);
        }
    }
    __syncthreads();
    if (S.nm < 0) {
        const int nl = pb ? 2 : s;
        if (tid < nl) levels[(int64_t)t * nl + tid] = 0.f;
        if (tid == 0) { status[t] |= OGQ_ST_INTERNAL; st->done = 1; }
        __threadfence();
        __syncthreads();
        return true;
    }
    // (the copies of the pass that just ended are complete unless it overflowed its region)
    const bool incomplete = round >= 2 && __ldcg(&st->overflow) != 0;
    const bool few = __syncthreads_and(tid >= S.nm || S.niv[tid].khi - S.niv[tid].klo < (1u << kRelBits)) && S.cand <= kSortN;
    if (round >= 2 && few && round_buf != nullptr && !incomplete) {
        const long long src_cnt = (long long)__ldcg(&st->cursor[round & 1]);
        if (src_cnt <= (enqueue ? kScanMax : kScanMaxAlone)) {
            finish_from_keys(st, t, pb, s, round_buf, (int)src_cnt, false, levels, status);
            return true;
        }
    }
    // prepare the next round: clear the cells it will use, publish the new intervals.  When the elements
    // inside the new intervals are few enough, the next pass only copies them and finish_sorted finishes
    // the tensor: no cells, no further solver pass.
    const bool compact_only = few && S.cand <= cap;
    const int ncells_next = S.niv[S.nm - 1].cellbase + S.niv[S.nm - 1].ncell;
    if (!compact_only) {
        for (int i = tid; i < ncells_next; i += nt) { gcnt[i] = 0u; glsum[i] = 0ull; }
    }
    if (tid < S.nm) st->iv[tid] = S.niv[tid];
    if (tid == 0) {
        st->m = S.nm;
        st->cand = S.cand;
        st->compact_only = compact_only ? 1 : 0;
        st->from_grad = incomplete ? 1 : 0;  // the next pass cannot read copies that were cut short
        st->overflow = 0;
        st->round = round + 1;
        st->arrive = 0;
        const int next = round + 1;
        st->cursor[next & 1] = 0ull;  // buffer the next round writes
        if (next == 3 && enqueue) {
            // work items of the round-3 kernel: slices of the copied keys, or of the tensor itself when
            // the copies were cut short
            const unsigned long long cntk = incomplete ? (unsigned long long)(S.view.n / 16) : __ldcg(&st->cursor[0]);
            unsigned ns = (unsigned)((cntk + kSliceElems - 1) / kSliceElems);
            if (ns < 1) ns = 1;
            if (ns > kMaxSlices) ns = kMaxSlices;
            st->expected = ns;
            const unsigned base = atomicAdd(nitems, ns);
            for (unsigned i = 0; i < ns; ++i) items[base + i] = make_int2(t, (int)i);
        }
    }
    __threadfence();
    __syncthreads();
    return false;
}

// Loads what solver_round needs of a tensor in round >= 2 back from its state.
__device__ __forceinline__ int solver_load(const TState* st, SolverShared& S, bool pb, int s)
{
    const int tid = threadIdx.x, m = __ldcg(&st->m);
    __syncthreads();
    if (tid < m) S.iv[tid] = st->iv[tid];
    if (!pb && tid >= 64 && tid - 64 < s) {
        const ExactLv& e = st->lv[tid - 64];
        LvInfo& l = S.lv[tid - 64];
        l.exact = e.exact; l.key = e.key;
        l.val = l.vlo = l.vhi = (double)sel_key_to_float(e.key);
        l.c_lt = e.c_lt; l.c_le = e.c_le; l.s_lt = e.s_lt; l.s_le = e.s_le;
    }
    if (tid == 0) {
        S.view.m = m;
        S.view.n = st->n;
        S.view.stot = st->stot;
    }
    return __ldcg(&st->round);
}

// ---------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------
struct SelArgs {
    const float* grad;
    const float* tau;  // per-tensor clipping thresholds, or null
    const int64_t* off;
    int T;
    int64_t total, chunk;  // chunk 0: shares of equal work (streamed_share)
    int first;             // the small tensors' launch is the first of the call
    int scheme, s;
    float* levels;
    int32_t* status;
    SelWs ws;
};

// One pass over grad[pb_, pe_) of tensor t with the tensor's current intervals (table and prefilter
// already built in tb): the values inside the intervals are copied to key buffer k (what fits the
// tensor's region) and, in mode 0, counted on the cells.
template <int NT>
__device__ __forceinline__ void grad_pass(const SelArgs& A, int t, int64_t tbeg, int64_t tend, int64_t pb_, int64_t pe_,
                                          int k, int mode)
{
    TState* st = A.ws.st + t;
    Round2Ctx& ctx = sel_table().ctx;
    if (threadIdx.x == 0) {
        ctx.dst = A.ws.buf[k] + sel_region(tbeg);
        ctx.cap = (unsigned long long)(sel_region(tend) - sel_region(tbeg));
        ctx.cursor = &st->cursor[k];
        ctx.overflow = &st->overflow;
        ctx.cursors = A.ws.gcnt + (size_t)t * kCells;
        ctx.clear = A.scheme == OGQ_BINGRAD_PB ? 0x7fffffffu : 0xffffffffu;
        ctx.mode = mode;
    }
    __syncthreads();
    // (round 2 itself goes against round 1's direction)
    if (A.tau) stream_round2<true, NT, false>(A.grad, pb_, pe_, __ldcg(A.tau + t));
    else stream_round2<false, NT, NT == kSelThreads>(A.grad, pb_, pe_, 0.f);
}

// Continues the rounds of one tensor on a single CTA until it is finished (the working set is
// tiny by then).  Called by the CTA that completed round >= 3.
__device__ void finish_alone(const SelArgs& A, int t)
{
    SolverShared& S = sel_state();
    Table& tb = sel_table();
    TState* st = A.ws.st + t;
    uint32_t* gcnt = A.ws.gcnt + (size_t)t * kCells;
    unsigned long long* glsum = A.ws.glsum + (size_t)t * kCells;
    uint32_t* hist = sel_hist();
    const int64_t tbeg = __ldg(A.off + t), tend = __ldg(A.off + t + 1);
    for (int guard = 0; guard < kMaxRounds; ++guard) {
        const int round = __ldcg(&st->round);
        const uint32_t* src = A.ws.buf[(round - 1) & 1];  // 16-byte aligned base; indices are absolute
        const int64_t cnt = (int64_t)__ldcg(&st->cursor[(round - 1) & 1]);
        const bool copy_only = st->compact_only != 0;
        __syncthreads();
        table_from_intervals(tb, st->iv, st->m);
        __syncthreads();
        if (!copy_only) zero_hist(hist, tb.ncells);
        __syncthreads();
        if (st->from_grad) {
            // the previous pass's copies did not fit: this pass reads the tensor itself again
            build_prefilter(tb, A.scheme == OGQ_BINGRAD_PB);
            grad_pass<kSolveThreads>(A, t, tbeg, tend, tbeg, tend, round & 1, copy_only);
        } else {
            Stager stg;
            stg.stage = sel_stage() + (threadIdx.x >> 5) * kStageCap;
            stg.dst = A.ws.buf[round & 1] + sel_region(tbeg);
            stg.cursor = &st->cursor[round & 1];
            stg.fill = 0;
            stream_piece(src, sel_region(tbeg), sel_region(tbeg) + cnt, tb, hist, hist + kCells, hist + 2 * kCells, stg, copy_only);
            stg.flush();
        }
        __syncthreads();
        if (copy_only) {
            __threadfence();
            __syncthreads();
            finish_sorted(st, t, A.scheme == OGQ_BINGRAD_PB, A.s, A.ws.buf[round & 1] + sel_region(tbeg), A.levels, A.status, round & 1);
            return;
        }
        flush_hist(hist, tb.ncells, gcnt, glsum);
        __threadfence();
        solver_load(st, S, A.scheme == OGQ_BINGRAD_PB, A.s);
        __syncthreads();
        if (solver_round(st, t, gcnt, glsum, A.scheme, A.s, A.levels, A.status, A.ws.nitems, A.ws.items,
                         A.ws.buf[round & 1] + sel_region(tbeg), false, sel_region(tend) - sel_region(tbeg), round))
            return;
    }
    if (threadIdx.x == 0) {
        A.status[t] |= OGQ_ST_ITER_CAP;
        st->done = 1;
    }
}

// The part [lo, hi) of the bucket that this CTA streams.  A piece of a tensor costs its elements and what its set-up and the
// flush of its cells take, as much as kPieceCost elements; tensors of at most kSmallN elements cost nothing.  Every CTA gets the same
// share of that sum.  (Equal chunks of the bucket instead: on the ResNet-50 bucket the CTAs of round 1 ended 23 to 40 us after its start, in
// the median 32, because some had three pieces and some mostly small tensors.)  Worked out by every CTA for itself, from the
// offsets alone, while the launch before is still running; with more than kMaxShared tensors chunks of the bucket are used.
constexpr int kPieceCost = 24576;
constexpr int kMaxShared = 8 * kSelThreads;
constexpr int kMinShare = 4 * kSelThreads * 4;  // elements per CTA of a small bucket: one trip of the streaming loops

__device__ __forceinline__ void streamed_share(const SelArgs& A, int64_t& lo, int64_t& hi)
{
    __shared__ long long sh_sum[kSelWarps], sh_at[2];
    if (A.chunk > 0) {
        lo = (int64_t)blockIdx.x * A.chunk;
        hi = (lo + A.chunk < A.total) ? lo + A.chunk : A.total;
        return;
    }
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = (A.T + kSelThreads - 1) / kSelThreads, t0 = min(tid * per, A.T), t1 = min(t0 + per, A.T);
    auto cost = [&](int t) -> long long {
        const long long n = __ldg(A.off + t + 1) - __ldg(A.off + t);
        return n <= kSmallN ? 0 : t > 0 ? n + kPieceCost : n;
    };
    long long own = 0;
    for (int t = t0; t < t1; ++t) own += cost(t);
    long long inc = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long nb = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += nb;
    }
    if (lane == 31) sh_sum[warp] = inc;
    if (tid < 2) sh_at[tid] = A.total;  // (a share that ends, or begins, behind the last streamed tensor)
    __syncthreads();
    const long long all = lane < kSelWarps ? sh_sum[lane] : 0;
    long long pos = warp_sum(lane < warp ? all : 0ll) + inc - own;
    const long long total = warp_sum(all), len = (total + gridDim.x - 1) / gridDim.x;
    for (int t = t0; t < t1; ++t) {
        const long long c = cost(t), tb = __ldg(A.off + t);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const long long x = ((long long)blockIdx.x + j) * len - pos;
            if (x >= 0 && x < c) {
                const long long lead = t > 0 ? kPieceCost : 0;
                sh_at[j] = x <= lead ? tb : max(tb, (tb + x - lead) & ~63ll);
            }
        }
        pos += c;
    }
    __syncthreads();
    lo = sh_at[0];
    hi = sh_at[1];
}

// Calls f(t, tensor_begin, tensor_end, piece_begin, piece_end) for the pieces of streamed tensors in [lo, hi), in ascending order
// or, when `down`, in descending order.  Called by all threads of a CTA; small tensors are passed over 32 at a time.
template <class F>
__device__ __forceinline__ void for_each_streamed(const SelArgs& A, int64_t lo, int64_t hi, F f, bool down)
{
    if (lo >= hi || A.T <= 0) return;
    const int lane = threadIdx.x & 31, dir = down ? -1 : 1;
    int t = find_tensor(A.off, A.T, down ? hi - 1 : lo);
    while (true) {
        const int mine = t + dir * lane;
        int64_t tb = 0, te = 0;
        bool in = false;
        if (mine >= 0 && mine < A.T) {
            tb = __ldg(A.off + mine);
            te = __ldg(A.off + mine + 1);
            in = tb < hi && te > lo;
        }
        const unsigned m = __ballot_sync(0xffffffffu, in && te - tb > kSmallN);
        if (!m) {
            if (!__shfl_sync(0xffffffffu, (int)(mine >= 0 && mine < A.T && (down ? te > lo : tb < hi)), 31)) return;
            t += 32 * dir;
            continue;
        }
        const int src = __ffs(m) - 1;
        const int64_t b = __shfl_sync(0xffffffffu, tb, src), e = __shfl_sync(0xffffffffu, te, src);
        t += dir * src;
        f(t, b, e, b > lo ? b : lo, e < hi ? e : hi);
        t += dir;
    }
}

// Anchor of a tensor's fine window in round 1: the largest binade among kSelThreads strided samples, plus two.  Called by every
// thread of a CTA, with this thread's sample; ends without a barrier (sh: kSelWarps values).
__device__ __forceinline__ float window_sample(const float* __restrict__ grad, int64_t tbeg, int64_t n)
{
    return __ldg(grad + tbeg + (int64_t)threadIdx.x * n / kSelThreads);
}
__device__ __forceinline__ int window_top(float sample, int* sh)
{
    int e = (int)((__float_as_uint(sample) >> 23) & 255u);
    if (e == 255) e = 0;
    e = __reduce_max_sync(0xffffffffu, e);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = e;
    __syncthreads();
    const int top = __reduce_max_sync(0xffffffffu, sh[threadIdx.x & (kSelWarps - 1)]) + 2;
    return min(max(top, kSelW), 255);  // binade 255 (Inf / NaN) always stays outside the fine window
}

// Clears what the passes over tensor t add to: one CTA per tensor.  Round 1 runs meanwhile and waits for it before it adds its cells.
__global__ void __launch_bounds__(kSelThreads) k_sel_prepare(SelArgs A)
{
    __shared__ int sh_i[kSelWarps];
    pdl_wait();
    pdl_launch_dependents();
    const int t = blockIdx.x;
    const int64_t tbeg = __ldg(A.off + t), n = __ldg(A.off + t + 1) - tbeg;
    if (t == 0 && threadIdx.x == 0) { A.ws.nitems[0] = 0u; A.ws.nitems[1] = 0u; }
    if (n <= kSmallN) return;
    const float sample = window_sample(A.grad, tbeg, n);
    const int ncells = A.scheme == OGQ_BINGRAD_PB ? kRound1Mag : kRound1Cells;
    uint4* cnt = reinterpret_cast<uint4*>(A.ws.gcnt + (size_t)t * kCells);
    uint4* sum = reinterpret_cast<uint4*>(A.ws.glsum + (size_t)t * kCells);
    for (int i = threadIdx.x; i < ncells / 4; i += kSelThreads) cnt[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int i = threadIdx.x; i < ncells / 2; i += kSelThreads) sum[i] = make_uint4(0u, 0u, 0u, 0u);
    const int hi_e = window_top(sample, sh_i);
    if (threadIdx.x == 0) {
        TState* st = A.ws.st + t;
        st->hi_e = hi_e;
        st->done = 0;
        st->kmin_inv = 0u;
        st->kmax = 0u;
        st->nonfinite = 0u;
        st->arrive = 0u;
        st->overflow = 0;
        st->from_grad = 0;
        st->compact_only = 0;
        st->cursor[0] = 0ull;
        st->cursor[1] = 0ull;
    }
}

// Flat CTAs: a share of the bucket each.  A piece of a tensor is streamed into the CTA's cells, which are then added to the
// tensor's global ones.  What it reads is the call's input, so it streams while the launch before still clears the global
// cells: that one has waited for everything earlier in the stream before it let this one start.
__global__ void __launch_bounds__(kSelThreads, kSelResident) k_sel_round1(SelArgs A)
{
    __shared__ int sh_top[kSelWarps];
    const bool pb = A.scheme == OGQ_BINGRAD_PB;
    uint32_t* hist = sel_hist();
    pdl_launch_dependents();
    uint32_t* packed_cells = sel_stage();
    const int ncells = pb ? kRound1Mag : kRound1Cells;
    int64_t lo, hi;
    streamed_share(A, lo, hi);
    for_each_streamed(A, lo, hi, [&](int t, int64_t tbeg, int64_t tend, int64_t pb_, int64_t pe_) {
        TState* st = A.ws.st + t;
        const float sample = window_sample(A.grad, tbeg, tend - tbeg);
        const float tau = A.tau ? __ldcg(A.tau + t) : 0.f;
        __syncthreads();
        zero_hist(hist, ncells);
        for (int i = threadIdx.x; i < kPackedCells; i += kSelThreads) packed_cells[i] = 0u;
        const int lo_e = window_top(sample, sh_top) - kSelW;  // (with a barrier)
        const bool clip = A.tau != nullptr;
        Round1Out r;
        if (pb) {
            if (clip) r = stream_round1<true, true>(A.grad, pb_, pe_, lo_e, tau);
            else r = stream_round1<true, false>(A.grad, pb_, pe_, lo_e, tau);
        } else {
            if (clip) r = stream_round1<false, true>(A.grad, pb_, pe_, lo_e, tau);
            else r = stream_round1<false, false>(A.grad, pb_, pe_, lo_e, tau);
        }
        pdl_wait();
        __syncthreads();
        flush_hist(hist, ncells, A.ws.gcnt + (size_t)t * kCells, A.ws.glsum + (size_t)t * kCells);
        // min / max / non-finite: one atomic per warp
        const uint32_t kmin = __reduce_min_sync(0xffffffffu, float_to_key(r.vmin));  // +Inf / -Inf when the
        const uint32_t kmax = __reduce_max_sync(0xffffffffu, float_to_key(r.vmax));  // thread saw nothing
        const bool anynf = __any_sync(0xffffffffu, r.nonfinite != 0u);
        if ((threadIdx.x & 31) == 0) {
            atomicMax(&st->kmin_inv, ~kmin);
            atomicMax(&st->kmax, kmax);
            if (anynf) atomicOr(&st->nonfinite, 1u);
        }
    }, A.tau != nullptr);
    pdl_wait();  // (a CTA without a piece: completion passes from kernel to kernel)
}

// ---------------------------------------------------------------------------
// The first solver pass: round 1's cells are the same for every tensor but for the position of the window, so
// their keys follow from their index.
// ---------------------------------------------------------------------------
struct Round1Cells {
    int lo_e;
    bool mag;  // cells of magnitudes only

    __device__ __forceinline__ int count() const { return mag ? kRound1Mag : kRound1Cells; }
    // keys of cell c: base, log2 of their number
    __device__ __forceinline__ uint32_t key(int c, int& sh) const
    {
        const bool neg = !mag && c < kRound1Mag;
        const int mi = mag ? c : neg ? kRound1Mag - 1 - c : c - kRound1Mag;
        const int k = mi - lo_e;
        const bool fine = k >= 0 && k < (kSelW << kSelM);
        sh = fine ? 23 - kSelM : 23;
        const uint32_t bits = fine ? ((uint32_t)lo_e << 23) + ((uint32_t)k << (23 - kSelM))
                                   : (uint32_t)(k < 0 ? mi : mi - (kSelW << kSelM) + kSelW) << 23;
        return neg ? 0x80000000u - bits - (1u << sh) : 0x80000000u + bits;
    }
    // exact sum of the cell's values: sel_cell_sum for these cells
    __device__ __forceinline__ double sum(int c, uint32_t cnt, unsigned long long lsum) const
    {
        const bool neg = !mag && c < kRound1Mag;
        const int mi = mag ? c : neg ? kRound1Mag - 1 - c : c - kRound1Mag;
        const int k = mi - lo_e;
        const bool fine = (unsigned)k < (unsigned)(kSelW << kSelM);
        const int e = fine ? lo_e + (k >> kSelM) : k < 0 ? mi : mi - (kSelW << kSelM) + kSelW;
        const uint32_t first = (e > 0 ? 1u << 23 : 0u) + (fine ? (uint32_t)(k & ((1 << kSelM) - 1)) << (23 - kSelM) : 0u);
        const uint32_t last = fine ? (1u << (23 - kSelM)) - 1u : (1u << 23) - 1u;
        // mantissas in units of 2^(max(e, 1) - 150); negative cells have their low bits mirrored
        const unsigned long long mant = (unsigned long long)cnt * first + (neg ? (unsigned long long)cnt * last - lsum : lsum);
        const double x = __ull2double_rn(mant) * __hiloint2double((max(e, 1) + 873) << 20, 0);
        return neg ? -x : x;
    }
};

// A level of the first pass: its value, or bounds of its value and the cells [sa, sb] that contain it.
struct Level1 {
    double vlo, vhi, s_lt, s_le;  // exact: value twice, sums before / up to it; else those of the whole range
    uint32_t c_lt, c_le;
    int exact, sa, sb;
};

struct __align__(16) Solve1Shared {
    Level1 lv[kMaxLv];
    uint32_t marks[(kRound1Cells + 31) / 32];
    int list[kCandCells], sorted[kCandCells];
    uint32_t starts[kCandCells / 32];   // which of the sorted candidate cells begin a run of neighbours
    int first[kMaxIv + 1], cells_at[kMaxIv + 1];
    int m, fail, runs;
    uint32_t cand, most;  // candidates, and those of the fullest cell
    int pb_a, pb_b;
};

constexpr size_t kOffCells1 = ((kRound1Cells + 8) * sizeof(double) + 15) / 16 * 16;  // prefix sums, then prefix counts, then the raw cells
constexpr size_t kOffRawSum1 = (kOffCells1 + (kRound1Cells + 8) * sizeof(uint32_t) + 15) / 16 * 16;
constexpr size_t kOffRawCnt1 = kOffRawSum1 + kRound1Cells * sizeof(unsigned long long);
static_assert(kOffRawCnt1 + kRound1Cells * sizeof(uint32_t) <= kIndexBytes, "the index of a small tensor takes more");

constexpr size_t kSolve1Bytes = kSolveBytes + sizeof(Solve1Shared);
__device__ __forceinline__ Solve1Shared& sel_state1() { return *reinterpret_cast<Solve1Shared*>(smem + kSolveBytes); }

// Q*(L, R) on round 1's cells by the 32 lanes of a warp; see warp_orq_solve for the bounds.
__device__ __noinline__ void solve1_level(int lo_e, double n, int q, int stride)
{
    const Round1Cells G{lo_e, false};
    const double* spre = reinterpret_cast<const double*>(smem);
    const uint32_t* cpre = reinterpret_cast<const uint32_t*>(smem + kOffCells1);
    Level1* out = sel_state1().lv + q;
    const int lane = threadIdx.x & 31;
    const bool upper = lane >= 16;
    const Level1 L = out[-stride], R = out[stride];
    const bool exact = L.exact && R.exact;
    if (exact && !(R.vlo > L.vlo)) {
        if (lane == 0) *out = L;
        __syncwarp();
        return;
    }
    const double floor_pos = (double)L.c_lt, ceil_pos = (double)R.c_le - 1.0;
    double p = upper ? ceil_pos : floor_pos;
    const double Cs = (double)(L.exact ? L.c_lt : L.c_le), Ce = (double)(R.exact ? R.c_le : R.c_lt);
    const double Ss = L.exact ? L.s_lt : L.s_le, Se = R.exact ? R.s_le : R.s_lt;
    const double cntM = Ce - Cs, sumM = Se - Ss;
    if (cntM >= 0.0 && R.vlo > L.vhi) {
        const double cntL = L.exact ? 0.0 : (double)(L.c_le - L.c_lt), cntR = R.exact ? 0.0 : (double)(R.c_le - R.c_lt);
        // (both brackets exact: both halves compute T = (sumM - L cntM) / (R - L))
        double num = fmax(sumM - (upper ? L.vhi : L.vlo) * cntM, 0.0);
        num = upper ? cntR * (R.vhi - R.vlo) - num : -(cntL * (L.vhi - L.vlo) + num);
        const double q = fp64_div(num, upper ? R.vhi - L.vhi : R.vlo - L.vlo);
        if (exact) {
            p = Ce - 1.0 - fmin(fmax(floor(-q), 0.0), cntM - 1.0);
        } else {
            const double delta = 2.0 + 1e-9 * n;
            const double g = ceil(Ce + q + (upper ? delta : -delta)) - 1.0;
            p = upper ? fmin(p, g) : fmax(p, g);
        }
    }
    p = fmin(fmax(p, floor_pos), ceil_pos);
    const double other = __shfl_xor_sync(0xffffffffu, p, 16);
    if (!upper) p = fmin(p, other);
    const uint32_t pos = __double2uint_rn(fmin(fmax(p, 0.0), n - 1.0));
    // the cells of the two ranks: the last whose prefix does not exceed the rank, by 32 probes in each of three steps
    const uint32_t pos_a = __shfl_sync(0xffffffffu, pos, 0), pos_b = __shfl_sync(0xffffffffu, pos, 16);
    constexpr int kStep1 = 161, kStep2 = 6;  // (an odd stride: different banks)
    static_assert(32 * kStep1 > kRound1Cells && 26 * kStep2 + 5 >= kStep1, "the probes reach every cell");
    const int nc = G.count();
    int sa = 0, sb = 0;
    auto probe = [&](int step, int probes) {
        const int ia = sa + (lane + 1) * step, ib = sb + (lane + 1) * step;
        const bool a = lane < probes && ia <= nc && cpre[min(ia, nc)] <= pos_a, b = lane < probes && ib <= nc && cpre[min(ib, nc)] <= pos_b;
        sa += step * __popc(__ballot_sync(0xffffffffu, a));
        sb += step * __popc(__ballot_sync(0xffffffffu, b));
    };
    probe(kStep1, 32);
    probe(kStep2, 26);
    probe(1, 5);
    const int slot = upper ? sb : sa;
    int sh;
    const uint32_t key = G.key(slot, sh);
    const double val = (double)sel_key_to_float(key + (upper ? (1u << sh) - 1u : 0u));
    const double vhi = __shfl_sync(0xffffffffu, val, 16);
    if (lane == 0) {
        out->exact = 0;
        out->vlo = val;
        out->vhi = vhi;
        out->sa = slot;
        out->sb = sb;
        out->c_lt = cpre[slot];
        out->s_lt = spre[slot];
        out->c_le = cpre[sb + 1];
        out->s_le = spre[sb + 1];
    }
    __syncwarp();
}

// One CTA per streamed tensor: prefix sums over round 1's cells, conservative cell ranges of the levels, every populated cell in
// them becomes an interval of round 2.
//   What bounds it: latency, 20,000 cycles of barriers, dependent loads and code that runs once (12,000 for BinGrad-pb).
__global__ void __launch_bounds__(kSolveThreads, 1) k_sel_solve1(SelArgs A)
{
    SolverShared& S = sel_state();
    Solve1Shared& Q = sel_state1();
    const bool pb = A.scheme == OGQ_BINGRAD_PB;
    const int nl = pb ? 2 : A.s, s = A.s;
    const int t = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t tbeg = __ldg(A.off + t), tend = __ldg(A.off + t + 1);
    const int64_t n = tend - tbeg;
    if (n <= kSmallN) {
        if (t == 0) pdl_wait();  // (one CTA at least: completion passes from kernel to kernel)
        return;
    }
    pdl_wait();
    pdl_launch_dependents();
    // (loads first, the decision what to do with them after)
    TState* st = A.ws.st + t;
    const uint32_t kmn = ~__ldcg(&st->kmin_inv), kmx = __ldcg(&st->kmax), nonfinite = __ldcg(&st->nonfinite);
    Round1Cells G;
    G.mag = pb;
    G.lo_e = __ldcg(&st->hi_e) - kSelW;
    const int ncells = G.count();
    uint32_t* gcnt = A.ws.gcnt + (size_t)t * kCells;
    unsigned long long* glsum = A.ws.glsum + (size_t)t * kCells;
    constexpr int kC = (kRound1Cells / 4 + kSolveThreads - 1) / kSolveThreads, kL = (kRound1Cells / 2 + kSolveThreads - 1) / kSolveThreads;
    uint4 c[kC];
    ulonglong2 l[kL];
#pragma unroll
    for (int u = 0; u < kC; ++u)
        if ((tid + u * kSolveThreads) * 4 < ncells) c[u] = __ldcg(reinterpret_cast<const uint4*>(gcnt) + tid + u * kSolveThreads);
#pragma unroll
    for (int u = 0; u < kL; ++u)
        if ((tid + u * kSolveThreads) * 2 < ncells) l[u] = __ldcg(reinterpret_cast<const ulonglong2*>(glsum) + tid + u * kSolveThreads);
    double* spre = reinterpret_cast<double*>(smem);
    uint32_t* cpre = reinterpret_cast<uint32_t*>(smem + kOffCells1);
    unsigned long long* raw_sum = reinterpret_cast<unsigned long long*>(smem + kOffRawSum1);
    uint32_t* raw_cnt = reinterpret_cast<uint32_t*>(smem + kOffRawCnt1);
    {
        if (tid < (kRound1Cells + 31) / 32) Q.marks[tid] = 0u;
        if (tid == 0) { Q.m = 0; Q.fail = 0; Q.runs = 0; Q.cand = 0u; Q.most = 0u; Q.pb_a = 0; Q.pb_b = 0; }
#pragma unroll
        for (int u = 0; u < kC; ++u)
            if ((tid + u * kSolveThreads) * 4 < ncells) reinterpret_cast<uint4*>(raw_cnt)[tid + u * kSolveThreads] = c[u];
#pragma unroll
        for (int u = 0; u < kL; ++u)
            if ((tid + u * kSolveThreads) * 2 < ncells) reinterpret_cast<ulonglong2*>(raw_sum)[tid + u * kSolveThreads] = l[u];
    }
    const bool bad = nonfinite != 0u, constant = !bad && !pb && kmn == kmx;
    if (bad || constant) {
        if (tid < nl) A.levels[(int64_t)t * nl + tid] = bad ? 0.f : sel_key_to_float(kmn);
        if (tid == 0) {
            A.status[t] = bad ? OGQ_ST_NONFINITE : OGQ_ST_CONSTANT;
            st->done = 1;
        }
        return;
    }
    __syncthreads();
    uint32_t total;
    double stot;
    {
        const int per = (ncells + kSolveThreads - 1) / kSolveThreads;
        const int c0 = tid * per < ncells ? tid * per : ncells, c1 = c0 + per < ncells ? c0 + per : ncells;
        uint32_t lc = 0u;
        double ls = 0.0;
#pragma unroll 1
        for (int c = c0; c < c1; ++c) {
            const uint32_t k = raw_cnt[c];
            double x = 0.0;
            if (k) x = G.sum(c, k, raw_sum[c]);
            spre[c] = x;
            lc += k;
            ls += x;
        }
        block_excl_scan(lc, ls, S, total, stot);
#pragma unroll 1
        for (int c = c0; c < c1; ++c) {
            const double x = spre[c];
            cpre[c] = lc;
            spre[c] = ls;
            lc += raw_cnt[c];
            ls += x;
        }
        // (the total is the last prefix: differences of prefixes, which decide where T falls on an integer, then carry
        // the rounding of one chain of additions)
        if (c0 < c1 && c1 == ncells) { cpre[ncells] = lc; spre[ncells] = ls; }
    }
    __syncthreads();
    stot = spre[ncells];
    if (tid >= 64 && tid - 64 < s && !pb) {
        const int q = tid - 64;
        Level1& l = Q.lv[q];
        l.exact = (q == 0 || q == s - 1) ? 1 : 0;
        l.vlo = l.vhi = (double)sel_key_to_float(q == 0 ? kmn : kmx);
        l.c_lt = 0u; l.s_lt = 0.0;
        l.c_le = q == 0 ? 0u : total; l.s_le = q == 0 ? 0.0 : stot;
        l.sa = l.sb = -1;
    }
    __syncthreads();
    const bool counted = (int64_t)total == n;
    int range_a = 0, range_b = -1;  // this warp's candidate cells
    if (counted && !pb) {
        static_assert(kSolveThreads / 32 >= kMaxLv - 1, "one warp per interior level");
#pragma unroll 1
        for (int stride = (s - 1) >> 1; stride >= 1; stride >>= 1) {
            const int q = warp;
            if (q < s - 1 && q >= stride && ((q - stride) & (2 * stride - 1)) == 0) {
                solve1_level(G.lo_e, (double)n, q, stride);
                if (!Q.lv[q].exact) {
                    range_a = Q.lv[q].sa;
                    range_b = Q.lv[q].sb;
                    if (range_a < 0 || range_a > range_b) Q.fail = 1;
                }
            }
            __syncthreads();
        }
    } else if (counted && stot > 0.0) {
        // bracket of the sign change of g(x) = x n - sum_{|v| >= x} |v|, evaluated at the lower edge of every cell
        int a = 0, b = 0;
#pragma unroll 1
        for (int c = tid; c < ncells; c += kSolveThreads) {
            int sh;
            const double x = (double)sel_key_to_float(G.key(c, sh));
            if (!(x < INFINITY)) continue;
            const double g = x * (double)n - (stot - spre[c]), eps = 1e-11 * (x * (double)n + stot);
            if (g < -eps) a = c;
            if (g <= eps) b = c;
        }
        a = __reduce_max_sync(0xffffffffu, a);
        b = __reduce_max_sync(0xffffffffu, b);
        if (lane == 0) { atomicMax(&Q.pb_a, a); atomicMax(&Q.pb_b, b); }
        __syncthreads();
        if (warp == 0) { range_a = Q.pb_a; range_b = max(Q.pb_a, Q.pb_b); }
    }
    // every populated cell of the ranges, once
#pragma unroll 1
    for (int base = range_a; base <= range_b; base += 32) {
        const int c = base + lane;
        const uint32_t k = c <= range_b ? cpre[c + 1] - cpre[c] : 0u, bit = 1u << (c & 31);
        const bool fresh = k && !(atomicOr(&Q.marks[c >> 5], bit) & bit);
        const uint32_t b = __ballot_sync(0xffffffffu, fresh), sum = __reduce_add_sync(0xffffffffu, fresh ? k : 0u);
        int i = 0;
        const uint32_t most = __reduce_max_sync(0xffffffffu, k);
        if (lane == 0 && b) {
            i = atomicAdd(&Q.m, __popc(b));
            atomicAdd(&Q.cand, sum);
            atomicMax(&Q.most, most);
        }
        i = __shfl_sync(0xffffffffu, i, 0) + __popc(b & ((1u << lane) - 1u));
        if (fresh && i < kCandCells) Q.list[i] = c;
    }
    __syncthreads();
    const int m = Q.m;
    if (tid == 0) {
        st->n = n;
        st->stot = stot;
        A.status[t] = 0;
    }
    if (!counted || Q.fail || (pb && !(stot > 0.0)) || m == 0) {
        // all magnitudes 0, an empty bracket (g is zero between two magnitudes), or an inconsistency
        const bool fail = !counted || !pb;
        if (pb) {
            const float b1 = fail || !(stot > 0.0) ? 0.f : (float)((stot - spre[Q.pb_a]) / (double)n);
            if (tid < 2) A.levels[2 * t + tid] = tid == 0 ? -b1 : b1;
        } else if (tid < s) {
            A.levels[(int64_t)t * s + tid] = 0.f;
        }
        if (tid == 0) {
            A.status[t] = fail ? OGQ_ST_INTERNAL : pb && !(stot > 0.0) ? OGQ_ST_CONSTANT : 0;
            st->done = 1;
        }
        return;
    }
    const uint32_t cand = Q.cand;
    bool compact_only = cand <= (uint32_t)kSortN && (int64_t)cand <= sel_region(tend) - sel_region(tbeg);
    // the candidate cells in order
    int my_rank = 0;
    uint32_t my_base = 0u;  // elements of those before, each rounded up to whole 128-bit words
    const bool mine = tid < m && m <= kCandCells;
    if (mine) {
        const int c = Q.list[tid];
#pragma unroll 4
        for (int j = 0; j < m; ++j) {
            const bool less = Q.list[j] < c;
            my_rank += less ? 1 : 0;
            if (cand > (uint32_t)kSortN && less) my_base += (cpre[Q.list[j] + 1] - cpre[Q.list[j]] + 3u) & ~3u;
        }
    }
    // Intervals of round 2: one per candidate cell when there are few, else one per run of neighbouring cells (of one
    // width); each gets the same share of the new cells.
    const bool single = m <= kMaxIv;
    int runs = m;
    if (!single) {
        if (mine) Q.sorted[my_rank] = Q.list[tid];
        __syncthreads();
        if (tid < kCandCells) {
            int s0, s1;
            bool start = false;
            if (tid < m && m <= kCandCells) {
                const uint32_t k1 = G.key(Q.sorted[tid], s1);
                const uint32_t k0 = tid > 0 ? G.key(Q.sorted[tid - 1], s0) : 0u;
                start = tid == 0 || s0 != s1 || k0 + (1u << s0) != k1;
            }
            const uint32_t w = __ballot_sync(0xffffffffu, start);
            if (lane == 0) { Q.starts[warp] = w; atomicAdd(&Q.runs, __popc(w)); }
        }
        __syncthreads();
        runs = m <= kCandCells ? Q.runs : kMaxIv + 1;
    }
    // More candidates than one CTA's index holds, but not more than the copies have room for: round 2 copies them in order of
    // these cells, and a level is selected among one cell's.
    const bool ordered = !pb && cand > (uint32_t)kSortN && (int64_t)cand + 3 * m <= sel_region(tend) - sel_region(tbeg) && runs <= kMaxIv;
    int r = runs <= kMaxIv && !ordered ? 31 - __clz(kCells / runs) : 0;
    bool fits = runs <= kMaxIv;
    int ncells_next = runs << r;
    if (!single && fits) {
        // position and length of every run, then halvings so that a run keeps to its share
        int id = -1;
        if (tid < m) {
            id = __popc(Q.starts[tid >> 5] & (0xffffffffu >> (31 - (tid & 31)))) - 1;
            for (int w = 0; w < (tid >> 5); ++w) id += __popc(Q.starts[w]);
            if ((Q.starts[tid >> 5] >> (tid & 31)) & 1u) Q.first[id] = tid;
        }
        if (tid == 0) Q.first[runs] = m;
        __syncthreads();
        const int share = kCells / runs;
        if (tid == 0) {
            int at = 0;
            for (int j = 0; j < runs; ++j) {
                const int len = Q.first[j + 1] - Q.first[j];
                Q.cells_at[j] = at;
                at += len <= share && !ordered ? len << (31 - __clz(share / len)) : len;
            }
            Q.cells_at[runs] = at;
        }
        __syncthreads();
        ncells_next = Q.cells_at[runs];
        fits = ncells_next <= kCells;
        bool narrow = true;
        if (fits && tid < runs) {
            const int len = Q.first[tid + 1] - Q.first[tid], c = Q.sorted[Q.first[tid]];
            int sh;
            Interval iv;
            iv.klo = G.key(c, sh);
            iv.khi = iv.klo + ((uint32_t)len << sh) - 1u;
            narrow = (unsigned long long)len << sh <= 1ull << kRelBits;
            const int rr = len <= share && !ordered ? 31 - __clz(share / len) : 0;
            iv.sh = sh - rr;
            iv.ncell = len << rr;
            iv.cellbase = Q.cells_at[tid];
            iv.pad = 0;
            iv.cbefore = cpre[c];
            iv.sbefore = spre[c];
            st->iv[tid] = iv;
        }
        compact_only = __syncthreads_and(narrow) && compact_only;
    }
    if (!fits) {
        // candidates scattered over too many cells: the general pass, which joins them up
        __syncthreads();
        if (tid < (pb ? 3 : 6)) S.iv[tid] = round1_interval(G.lo_e + kSelW, pb, tid);
        if (tid >= 64 && tid - 64 < s) {
            LvInfo& l = S.lv[tid - 64];
            l.exact = (tid == 64 || tid - 64 == s - 1) ? 1 : 0;
            l.key = tid == 64 ? kmn : kmx;
            l.val = l.vlo = l.vhi = (double)sel_key_to_float(l.key);
            l.c_lt = 0; l.s_lt = 0.0; l.c_le = 0; l.s_le = 0.0;
        }
        if (tid == 0) { S.view.m = pb ? 3 : 6; S.view.n = n; S.view.stot = 0.0; }
        solver_round(st, t, gcnt, glsum, A.scheme, s, A.levels, A.status, A.ws.nitems, A.ws.items, nullptr, false, sel_region(tend) - sel_region(tbeg), 1);
        return;
    }
    if (single && mine) {
        const int c = Q.list[tid];
        Interval iv;
        int sh;
        iv.klo = G.key(c, sh);
        iv.khi = iv.klo + ((1u << sh) - 1u);
        iv.sh = sh - r;
        iv.ncell = 1 << r;
        iv.cellbase = my_rank << r;
        iv.pad = 0;
        iv.cbefore = cpre[c];
        iv.sbefore = spre[c];
        st->iv[my_rank] = iv;
    }
    if (!pb && tid >= 64 && tid - 64 < s) {
        const Level1& l = Q.lv[tid - 64];
        ExactLv& e = st->lv[tid - 64];
        e.exact = l.exact;
        e.key = float_to_key((float)l.vlo);
        e.c_lt = l.c_lt; e.c_le = l.c_le; e.s_lt = l.s_lt; e.s_le = l.s_le;
    }
    if (ordered) {
        if (mine) {
            const int c = Q.list[tid];
            CandCell x;
            x.sbefore = spre[c];
            x.cbefore = cpre[c];
            x.n = cpre[c + 1] - cpre[c];
            x.klo = G.key(c, x.sh);
            x.base = my_base;
            x.pad = 0;
            reinterpret_cast<CandCell*>(glsum)[my_rank] = x;
            gcnt[tid] = 0u;
        }
        if (tid == 0 && Q.most > (uint32_t)kCellsAlone) A.ws.items[(size_t)A.T * kMaxSlices - 1 - atomicAdd(A.ws.nitems + 1, 1u)].x = t;
    } else if (!compact_only) {
        for (int i = tid; i < ncells_next; i += kSolveThreads) { gcnt[i] = 0u; glsum[i] = 0ull; }
    }
    if (tid == 96) {
        if (ordered) st->arrive = Q.most;
        st->m = runs;
        st->cand = cand;
        if (ordered) st->expected = (unsigned)m;
        st->compact_only = ordered ? (Q.most > (uint32_t)kCellsAlone ? kOrderedLarger : kOrdered) : compact_only ? kCompact : kCounted;
        st->round = 2;
    }
}

__global__ void __launch_bounds__(kSelThreads, kSelResident) k_sel_round2(SelArgs A)
{
    Table& tb = sel_table();
    const bool pb = A.scheme == OGQ_BINGRAD_PB;
    uint32_t* hist = sel_hist();
    int64_t lo, hi;
    streamed_share(A, lo, hi);
    pdl_wait();
    pdl_launch_dependents();
    // Second pass over a piece: builds the tensor's interval table and prefilter, clears the CTA's cells,
    // copies the values inside the intervals and counts them on the finer cells (unless they already fit
    // one sort), adds the cells to the tensor's global ones.
    const bool down = A.tau == nullptr;  // against round 1's direction
    for_each_streamed(A, lo, hi, [&](int t, int64_t tbeg, int64_t tend, int64_t pb_, int64_t pe_) {
        TState* st = A.ws.st + t;
        if (__ldcg(&st->done)) return;  // settled in round 1
        __syncthreads();
        table_from_intervals(tb, st->iv, __ldcg(&st->m));
        __syncthreads();
        build_prefilter(tb, pb);
        const int mode = min(__ldcg(&st->compact_only), kOrdered);
        if (mode == 0) zero_hist(hist, tb.ncells);
        if (mode == 2) {
            const CandCell* cells = reinterpret_cast<const CandCell*>(A.ws.glsum + (size_t)t * kCells);
            const int m = (int)__ldcg(&st->expected);
            for (int i = threadIdx.x; i < kCandCells; i += kSelThreads) {
                sel_partition().base[i] = i < m ? __ldcg(&cells[i].base) : 0u;
                sel_partition().cnt[i] = 0u;
            }
            if (threadIdx.x == 0) tb.cta_fill = 0;
        }
        __syncthreads();
        grad_pass<kSelThreads>(A, t, tbeg, tend, pb_, pe_, 0, mode);
        if (mode == 2) partition_flush();
        __syncthreads();
        if (mode == 0) flush_hist(hist, tb.ncells, A.ws.gcnt + (size_t)t * kCells, A.ws.glsum + (size_t)t * kCells);
    }, down);
}

// ---------------------------------------------------------------------------
// ORQ tensors with more candidates than one CTA's index holds: their keys lie in order of round 1's candidate cells, whose
// exact counts and sums are known.  The exact rank of a level, known when its two brackets are, tells the cell; the level is
// selected among that cell's keys alone.  Cells of up to kCellsAlone keys: by one CTA, a group of its warps on every level of a depth of Algorithm
// 1, by counts on some of the keys' bits at a time, the upper ones first.
//   What bounds it: latency, 6000 cycles a depth for small cells.  A cluster (tensor_from_cells) takes 20,000 for its barriers and for what its CTAs
// read from one another's shared memory, whatever the number of keys: 1.2 M elements of 17 levels 82 -> 57 us.
// ---------------------------------------------------------------------------
constexpr int kGroups = 8;         // levels of a depth
constexpr int kGroupThreads = 256; // of a level's group, at most, where cells are small
constexpr int kRest = 32;          // keys that are left to one warp

struct GroupSelect {
    int cell, open;       // the rank's cell, -1: none has it; whether there is a rank (the brackets differ)
    uint32_t rank;        // of the level
    uint32_t bin, below, own;
    uint32_t listed, list[kRest];
    uint32_t warp_n[kSolveThreads / 32];
    unsigned long long warp_sum[kSolveThreads / 32];
};

struct __align__(16) CellGroups {
    LvInfo lv[kMaxLv];
    GroupSelect group[kGroups];
    uint32_t bins[kGroups * 2 * (kSolveThreads / kGroups)];  // two a thread
    int fail;
    CandCell cells[kCandCells];
};
static_assert(sizeof(CellGroups) <= kIndexBytes, "fits the solver's shared memory");
__device__ __forceinline__ CellGroups& cell_groups() { return *reinterpret_cast<CellGroups*>(smem); }

// The cells of tensor t into `cells`, by every thread of the CTA; those beyond the last begin behind everything.  The caller synchronises.
__device__ __forceinline__ void cells_load(const SelArgs& A, const TState* st, int t, CandCell* cells)
{
    static_assert(kCandCells <= kSolveThreads, "a thread per candidate cell");
    if (threadIdx.x < kCandCells) {
        CandCell x = reinterpret_cast<const CandCell*>(A.ws.glsum + (size_t)t * kCells)[threadIdx.x];
        if ((int)threadIdx.x >= (int)__ldcg(&st->expected)) {
            x.cbefore = 0xffffffffu;
            x.n = 0u;
        }
        cells[threadIdx.x] = x;
    }
}

// Level q between levels q - stride and q + stride, by the `threads` threads (a power of two) of group g, which all call this; a barrier
// of the caller's ends it.  keys: the tensor's copied keys.
__device__ __noinline__ void level_by_group(int q, int stride, int g, int threads, const uint32_t* keys)
{
    CellGroups& Q = cell_groups();
    GroupSelect& X = Q.group[g];
    const int gt = (int)threadIdx.x & (threads - 1), lane = gt & 31, warp = gt >> 5, warps = threads >> 5;
    uint32_t* bins = Q.bins + g * 2 * threads;
    const int bin_bits = 32 - __clz(threads);
    auto sync = [&]() { asm volatile("bar.sync %0, %1;" :: "r"(g + 1), "r"(threads) : "memory"); };
    if (warp == 0) {
        const LvInfo &L = Q.lv[q - stride], &R = Q.lv[q + stride];
        const double width = R.val - L.val, nseg = (double)((uint32_t)R.c_le - (uint32_t)L.c_lt);
        const bool open = width > 0.0;
        const uint32_t p = open ? (uint32_t)R.c_le - 1u - (uint32_t)fmin(fmax(floor_of_t(R.s_le, L.s_lt, L.val, width, nseg), 0.0), nseg - 1.0) : 0u;
        // the last cell that begins at or before rank p
        constexpr int kStep = kCandCells / 32;
        int c = __popc(__ballot_sync(0xffffffffu, Q.cells[lane * kStep].cbefore <= p)) - 1;
        if (c >= 0) c = c * kStep + __popc(__ballot_sync(0xffffffffu, lane < kStep && Q.cells[c * kStep + (lane & (kStep - 1))].cbefore <= p)) - 1;
        const bool in = open && c >= 0 && p - Q.cells[max(c, 0)].cbefore < Q.cells[max(c, 0)].n;
        if (lane == 0) {
            X.cell = in ? c : -1;
            X.open = open ? 1 : 0;
            X.rank = p;
            X.listed = 0u;
        }
    }
    reinterpret_cast<uint2*>(bins)[gt] = make_uint2(0u, 0u);
    sync();
    if (X.cell < 0) {
        if (gt == 0) {
            Q.lv[q] = Q.lv[q - stride];
            if (X.open) Q.fail = 1;  // no candidate cell holds the rank: an inconsistency
        }
        return;
    }
    const CandCell& cell = Q.cells[X.cell];
    const int n = (int)cell.n;
    const uint4* src = reinterpret_cast<const uint4*>(keys + cell.base);
    uint32_t k = X.rank - cell.cbefore, prefix = 0u, below = 0u;
    int rem = cell.sh, own = n;  // bits that are still open; keys that share the others
    unsigned long long sum = 0ull;
    auto each = [&](auto f) {
        constexpr int kCols = 2;  // loads in flight
#pragma unroll 1
        for (int i0 = gt; 4 * i0 < n; i0 += kCols * threads) {
            uint4 x[kCols];
#pragma unroll
            for (int u = 0; u < kCols; ++u)
                if (4 * (i0 + u * threads) < n) x[u] = __ldcg(src + i0 + u * threads);
#pragma unroll
            for (int u = 0; u < kCols; ++u) {
                const int left = n - 4 * (i0 + u * threads);
                if (left > 0) f(x[u].x);
                if (left > 1) f(x[u].y);
                if (left > 2) f(x[u].z);
                if (left > 3) f(x[u].w);
            }
        }
    };
#pragma unroll 1
    while (rem > 0 && own > kRest) {
        const int bits = min(rem, bin_bits), shift = rem - bits;
        each([&](uint32_t x) {
            if (x >> rem == prefix) atomicAdd(bins + ((x >> shift) & ((1u << bits) - 1u)), 1u);
        });
        sync();
        const uint2 c = reinterpret_cast<const uint2*>(bins)[gt];
        uint32_t inc = c.x + c.y;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t nb = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += nb;
        }
        if (lane == 31) X.warp_n[warp] = inc;
        reinterpret_cast<uint2*>(bins)[gt] = make_uint2(0u, 0u);  // (for the next bits)
        sync();
        const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? X.warp_n[lane] : 0u) + inc - (c.x + c.y);
        if (before <= k && k - before < c.x + c.y) {
            const bool second = k - before >= c.x;
            X.bin = 2u * (uint32_t)gt + (second ? 1u : 0u);
            X.below = before + (second ? c.x : 0u);
            X.own = second ? c.y : c.x;
        }
        sync();
        const uint32_t next = prefix << bits | X.bin;
        own = (int)X.own;
        below += X.below;
        k -= X.below;
        if (stride > 1)
            each([&](uint32_t x) {
                if (x >> shift < next && x >> rem == prefix) sum += x;
            });
        prefix = next;
        rem = shift;
    }
    if (rem > 0)  // a few keys, for one warp
        each([&](uint32_t x) {
            if (x >> rem == prefix) X.list[atomicAdd(&X.listed, 1u)] = x;
        });
    sum = (unsigned long long)warp_sum((long long)sum);
    if (lane == 0) X.warp_sum[warp] = sum;
    sync();
    if (warp != 0) return;
    sum = (unsigned long long)warp_sum(lane < warps ? (long long)X.warp_sum[lane] : 0ll);
    uint32_t rel = prefix, lt = 0u, eq = (uint32_t)own;
    if (rem > 0) {  // the k-th of them
        rel = lane < own ? X.list[lane] : 0xffffffffu;
        eq = 0u;
        uint32_t smaller = 0u;
#pragma unroll 4
        for (int j = 0; j < own; ++j) {
            const uint32_t x = X.list[j];
            if (x < rel) { ++lt; smaller += x; }
            eq += x == rel ? 1u : 0u;
        }
        const int at = (__ffs(__ballot_sync(0xffffffffu, lane < own && lt <= k && k - lt < eq)) - 1) & 31;
        rel = __shfl_sync(0xffffffffu, rel, at);
        lt = __shfl_sync(0xffffffffu, lt, at);
        eq = __shfl_sync(0xffffffffu, eq, at);
        sum += __shfl_sync(0xffffffffu, smaller, at);
    }
    if (lane == 0) {
        LvInfo& o = Q.lv[q];
        lt += below;
        o.val = (double)sel_key_to_float(cell.klo + rel);
        o.c_lt = (long long)cell.cbefore + lt;
        o.c_le = o.c_lt + eq;
        o.s_lt = cell.sbefore + sel_cell_sum(cell.klo, cell.sh, lt, sum);  // (of the last depth's levels nobody asks)
        o.s_le = o.s_lt + o.val * (double)eq;
    }
}

// The levels of tensor t, by one CTA.
__device__ __forceinline__ void levels_from_cells(const SelArgs& A, TState* st, int t, const uint32_t* keys, int most_threads)
{
    CellGroups& Q = cell_groups();
    const int tid = threadIdx.x, s = A.s;
    __syncthreads();
    cells_load(A, st, t, Q.cells);
    if (tid >= kCandCells && tid - kCandCells < s) {
        const ExactLv& e = st->lv[tid - kCandCells];
        LvInfo& l = Q.lv[tid - kCandCells];
        l.val = (double)sel_key_to_float(e.key);
        l.c_lt = e.c_lt; l.c_le = e.c_le; l.s_lt = e.s_lt; l.s_le = e.s_le;
    }
    if (tid == kSolveThreads - 1) Q.fail = 0;
    __syncthreads();
#pragma unroll 1
    for (int stride = (s - 1) >> 1; stride >= 1; stride >>= 1) {
        const int levels = (s - 1) / (2 * stride), threads = min(kSolveThreads / levels, most_threads), g = tid / threads;
        if (g < levels) level_by_group(stride * (2 * g + 1), stride, g, threads, keys);
        __syncthreads();
    }
    if (tid < s) A.levels[(int64_t)t * s + tid] = Q.fail ? 0.f : (float)Q.lv[tid].val;
    if (tid == 0) {
        if (Q.fail) A.status[t] |= OGQ_ST_INTERNAL;
        st->done = 1;
    }
    __syncthreads();
}

// Small tensors let what follows be launched while they are worked on, in buckets of up to this size: 100 tensors of 16,000 elements, nine
// levels, 33.9 us instead of 36.4, 20 of 9000 and one of 200,000 values 46 instead of 48.  Larger ones, whose round 3 has work, get slower (40 M
// elements in 120 tensors, BinGrad-pb: 200 instead of 191).
constexpr int64_t kEarlyN = 1 << 24;

// What follows round 2, one CTA per tensor: the finish from the copied keys when round 2 only copied, else a solver pass and
// work items of the round-3 kernel.  Small tensors are solved here, from the call's input alone, so before the rounds are waited
// for: in the first solver pass, whose launch they made longer (ResNet-50 bucket: 161 CTAs on 148 SMs, 21 us instead of 10), they
// stood in the way of the streamed tensors.
__global__ void __launch_bounds__(kSolveThreads, 1) k_sel_solve2(SelArgs A)
{
    if (A.first) pdl_wait();
    const int t = blockIdx.x;
    SolverShared& S = sel_state();
    const int64_t tbeg = __ldg(A.off + t), tend = __ldg(A.off + t + 1);
    const int64_t n = tend - tbeg;
    if (n <= kSmallN) {
        // (what follows waits for this whole launch, and with it for the CTAs that do wait)
        if (A.total < kEarlyN) pdl_launch_dependents();
        const bool pb = A.scheme == OGQ_BINGRAD_PB;
        const int nl = pb ? 2 : A.s;
        if (n <= 0) {
            if ((int)threadIdx.x < nl) A.levels[(int64_t)t * nl + threadIdx.x] = 0.f;
            if (threadIdx.x == 0) A.status[t] = OGQ_ST_EMPTY;
        } else {
            small_tensor(A.grad + tbeg, (int)n, t, pb, A.s, A.levels, A.status, A.tau ? __ldcg(A.tau + t) : __int_as_float(0x7f800000));
        }
        if (t == 0) pdl_wait();  // (one CTA at least: completion passes from kernel to kernel)
        return;
    }
    pdl_wait();
    pdl_launch_dependents();
    TState* st = A.ws.st + t;
    const int done = __ldcg(&st->done), compact_only = __ldcg(&st->compact_only);
    const long long cand = __ldcg(&st->cand), src_cnt = (long long)__ldcg(&st->cursor[0]);
    finish_load(st, A.scheme == OGQ_BINGRAD_PB, A.s, S);  // (all loads in one go, the decision what to do with them after)
    if (done || compact_only == kOrderedLarger) return;
    if (compact_only == kOrdered) {
        const int most = (int)__ldcg(&st->arrive);
        if (most > kCellsBeside && __ldcg(A.ws.nitems + 1) > 0u) {
            if (threadIdx.x == 0) A.ws.items[(size_t)A.T * kMaxSlices - 1 - atomicAdd(A.ws.nitems + 1, 1u)].x = t;
            return;
        }
        levels_from_cells(A, st, t, A.ws.buf[0] + sel_region(tbeg), most > kCellsBeside ? kSolveThreads : kGroupThreads);
        return;
    }
    if (compact_only == kCompact) {
        finish_from_keys(st, t, A.scheme == OGQ_BINGRAD_PB, A.s, A.ws.buf[0] + sel_region(tbeg), (int)min(src_cnt, cand), true,
                         A.levels, A.status);
        return;
    }
    const int round = solver_load(st, S, A.scheme == OGQ_BINGRAD_PB, A.s);
    solver_round(st, t, A.ws.gcnt + (size_t)t * kCells, A.ws.glsum + (size_t)t * kCells, A.scheme, A.s, A.levels, A.status,
                 A.ws.nitems, A.ws.items, A.ws.buf[0] + sel_region(tbeg), true, sel_region(tend) - sel_region(tbeg), round);
}

// ---------------------------------------------------------------------------
// Tensors with more candidates than one CTA's index holds: their keys lie in order of round 1's candidate cells, whose
// exact counts and sums are known.  The exact rank of a level, known when its two brackets are, tells the cell; the level is
// selected among that cell's keys alone, by counts on their upper and then on their lower bits.  A cluster per tensor;
// the CTAs share out the levels of a depth of Algorithm 1, and where there are fewer levels than CTAs, the keys of a cell.
//   What bounds it: the latency of a depth, two reads of a cell's keys (80,000 of 50 M values) and three cluster barriers.
// It takes the place of a finer histogram in round 2, a solver pass on it and a third round.
// ---------------------------------------------------------------------------
constexpr int kCluster = 8;     // CTAs: the levels of the last depth of 17
constexpr int kUpperBits = 11;  // of a key, in the first count

struct __align__(16) CellSelect {
    uint32_t upper[1 << kUpperBits], lower[1 << (kCellBits - kUpperBits)];
    LvInfo lv[kMaxLv];
    unsigned long long part[32], sum;  // of the keys below the upper bits' range, this CTA's share
    uint32_t warp_n[32];
    int cell, open, fail;    // the rank's cell, -1: none has it; whether there is a rank (the brackets differ)
    uint32_t rank;           // of the level
    uint32_t bin, below, n;  // what bin_of_rank found
    CandCell cells[kCandCells];
};
static_assert(sizeof(CellSelect) <= kIndexBytes, "fits the solver's shared memory");

__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_address(const void* p, int rank)
{
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm("mapa.shared::cluster.u32 %0, %0, %1;" : "+r"(a) : "r"(rank));
    return a;
}

// The bin that holds rank r, from the counts of `group` CTAs from rank `first` on: to Q.bin, Q.below (elements before it) and
// Q.n (its own).  PER: bins of a thread; c: their counts on return.  Called by every thread; ends with a barrier.
template <int PER>
__device__ __forceinline__ void bin_of_rank(CellSelect& Q, const uint32_t* bins, int nbins, int first, int group, uint32_t r, uint32_t (&c)[PER])
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll
    for (int j = 0; j < PER; ++j) c[j] = 0u;
    if (tid * PER < nbins) {
        static_assert(PER % 2 == 0, "two bins a load");
        uint32_t x[kCluster][PER];
#pragma unroll
        for (int g = 0; g < kCluster; ++g) {  // (all loads before the first is used: one at a time, this took 13,000 cycles)
#pragma unroll
            for (int j = 0; j < PER; j += 2) {
                x[g][j] = x[g][j + 1] = 0u;
                if (g < group)
                    asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];" : "=r"(x[g][j]), "=r"(x[g][j + 1])
                                 : "r"(cluster_address(bins + tid * PER + j, first + g)));
            }
        }
#pragma unroll
        for (int g = 0; g < kCluster; ++g)
#pragma unroll
            for (int j = 0; j < PER; ++j) c[j] += x[g][j];
    }
    uint32_t own = 0u;
#pragma unroll
    for (int j = 0; j < PER; ++j) own += c[j];
    uint32_t inc = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t nb = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += nb;
    }
    if (lane == 31) Q.warp_n[warp] = inc;
    __syncthreads();
    uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? Q.warp_n[lane] : 0u) + inc - own;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        if (before <= r && r - before < c[j]) { Q.bin = (uint32_t)(tid * PER + j); Q.below = before; Q.n = c[j]; }
        before += c[j];
    }
    __syncthreads();
}

// Sum over the CTA's threads, valid in all of them.
__device__ __forceinline__ unsigned long long cta_sum(CellSelect& Q, unsigned long long x)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    x = (unsigned long long)warp_sum((long long)x);
    if (lane == 0) Q.part[warp] = x;
    __syncthreads();
    return (unsigned long long)warp_sum((long long)Q.part[lane]);
}

// Tensor t by the CTAs of a cluster, all of which call this.
__device__ __noinline__ void tensor_from_cells(const SelArgs& A, int t, int rank)
{
    CellSelect& Q = *reinterpret_cast<CellSelect*>(smem);
    const int tid = threadIdx.x, s = A.s;
    TState* st = A.ws.st + t;
    const CandCell* cells = reinterpret_cast<const CandCell*>(A.ws.glsum + (size_t)t * kCells);
    const uint32_t* keys = A.ws.buf[0] + sel_region(__ldg(A.off + t));
    uint32_t cb = 0xffffffffu, cn = 0u;  // the candidate cell of this thread
    static_assert(kCandCells <= kSolveThreads, "a thread per candidate cell");
    if (tid < kCandCells) {
        const CandCell x = cells[tid];  // (those beyond the last are not cells)
        if (tid < (int)__ldcg(&st->expected)) {
            Q.cells[tid] = x;
            cb = x.cbefore;
            cn = x.n;
        }
    }
    if (tid < s) {
        const ExactLv& e = st->lv[tid];
        LvInfo& l = Q.lv[tid];
        l.val = (double)sel_key_to_float(e.key);
        l.c_lt = e.c_lt; l.c_le = e.c_le; l.s_lt = e.s_lt; l.s_le = e.s_le;
    }
    if (tid == 0) Q.fail = 0;
    cluster_sync_all();  // (nobody writes into a CTA that is not here yet)
#pragma unroll 1
    for (int stride = (s - 1) >> 1; stride >= 1; stride >>= 1) {
        const int group = kCluster * 2 * stride / (s - 1), first = rank / group * group;  // the CTAs that share this one's level
        const int q = stride * (2 * (rank / group) + 1);
        const LvInfo &L = Q.lv[q - stride], &R = Q.lv[q + stride];
        if (tid < 32) {  // (by one warp: the fp64 unit is the bottleneck when all compute the same)
            const double width = R.val - L.val, nseg = (double)((uint32_t)R.c_le - (uint32_t)L.c_lt);
            const bool open = width > 0.0;
            if (tid == 0) {
                Q.cell = -1;
                Q.open = open ? 1 : 0;
                Q.rank = open ? (uint32_t)R.c_le - 1u - (uint32_t)fmin(fmax(floor_of_t(R.s_le, L.s_lt, L.val, width, nseg), 0.0), nseg - 1.0) : 0u;
            }
        }
        __syncthreads();
        const bool open = Q.open != 0;
        const uint32_t p = Q.rank;
        if (open && cb <= p && p - cb < cn) Q.cell = tid;
        __syncthreads();
        const int c = Q.cell;
        // this CTA's share of the cell's keys
        int share = 0, sh = kUpperBits;
        const uint4* src = nullptr;
        CandCell cell = {};
        if (c >= 0) {
            cell = Q.cells[c];
            sh = cell.sh;
            const int per = (((int)cell.n + group - 1) / group + 3) & ~3, begin = min((rank - first) * per, (int)cell.n);
            share = min(per, (int)cell.n - begin);
            src = reinterpret_cast<const uint4*>(keys + cell.base + begin);
        }
        const int low = sh - kUpperBits;  // lower bits
        auto each = [&](auto f) {
            constexpr int kCols = 4;  // loads in flight
#pragma unroll 1
            for (int i0 = tid; 4 * i0 < share; i0 += kCols * kSolveThreads) {
                uint4 k[kCols];
#pragma unroll
                for (int u = 0; u < kCols; ++u)
                    if (4 * (i0 + u * kSolveThreads) < share) k[u] = __ldcg(src + i0 + u * kSolveThreads);
#pragma unroll
                for (int u = 0; u < kCols; ++u) {
                    const int left = share - 4 * (i0 + u * kSolveThreads);
                    if (left > 0) f(k[u].x);
                    if (left > 1) f(k[u].y);
                    if (left > 2) f(k[u].z);
                    if (left > 3) f(k[u].w);
                }
            }
        };
        for (int i = tid; i < 1 << kUpperBits; i += kSolveThreads) Q.upper[i] = 0u;
        for (int i = tid; i < 1 << low; i += kSolveThreads) Q.lower[i] = 0u;
        __syncthreads();
        each([&](uint32_t k) { atomicAdd(&Q.upper[(k >> low) & ((1u << kUpperBits) - 1u)], 1u); });
        cluster_sync_all();
        uint32_t below = 0u, bin = 0u;
        if (c >= 0) {
            uint32_t n2[(1 << kUpperBits) / kSolveThreads];
            bin_of_rank(Q, Q.upper, 1 << kUpperBits, first, group, p - cell.cbefore, n2);
            below = Q.below;
            bin = Q.bin;
        }
        unsigned long long sum = 0ull;
        each([&](uint32_t k) {
            if (k >> low == bin) atomicAdd(&Q.lower[k & ((1u << low) - 1u)], 1u);
            else if (k >> low < bin) sum += k;
        });
        sum = cta_sum(Q, sum);
        if (tid == 0) Q.sum = sum;
        cluster_sync_all();
        if (rank == first) {
            uint32_t n_lt = 0u;
            if (c >= 0) {
                constexpr int kPer = (1 << (kCellBits - kUpperBits)) / kSolveThreads;
                uint32_t n4[kPer];
                bin_of_rank(Q, Q.lower, 1 << low, first, group, p - cell.cbefore - below, n4);
                // the keys of the range that are smaller, from their counts
                sum = 0ull;
#pragma unroll
                for (int j = 0; j < kPer; ++j)
                    if ((uint32_t)(tid * kPer + j) < Q.bin) sum += (unsigned long long)n4[j] * ((bin << low) + (uint32_t)(tid * kPer + j));
                if (tid < group) {
                    unsigned long long x;
                    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(x) : "r"(cluster_address(&Q.sum, first + tid)));
                    sum += x;
                }
                sum = cta_sum(Q, sum);
                n_lt = below + Q.below;
            }
            if (tid < kCluster) {
                LvInfo o = L;
                if (c >= 0) {
                    o.val = (double)sel_key_to_float(cell.klo + (bin << low) + Q.bin);
                    o.c_lt = (long long)cell.cbefore + n_lt;
                    o.c_le = o.c_lt + Q.n;
                    o.s_lt = cell.sbefore + sel_cell_sum(cell.klo, sh, n_lt, sum);
                    o.s_le = o.s_lt + o.val * (double)Q.n;
                }
                const uint32_t to = cluster_address(&Q.lv[q], tid);
                auto put = [&](size_t at, auto x) {
                    asm volatile("st.shared::cluster.b64 [%0], %1;" :: "r"(to + (uint32_t)at), "l"(x) : "memory");
                };
                put(offsetof(LvInfo, val), __double_as_longlong(o.val));
                put(offsetof(LvInfo, c_lt), o.c_lt);
                put(offsetof(LvInfo, c_le), o.c_le);
                put(offsetof(LvInfo, s_lt), __double_as_longlong(o.s_lt));
                put(offsetof(LvInfo, s_le), __double_as_longlong(o.s_le));
                if (c < 0 && open)  // no candidate cell holds the rank: an inconsistency
                    asm volatile("st.shared::cluster.b32 [%0], %1;" :: "r"(cluster_address(&Q.fail, tid)), "r"(1) : "memory");
            }
        }
        cluster_sync_all();
    }
    if (rank == 0) {
        if (tid < s) A.levels[(int64_t)t * s + tid] = Q.fail ? 0.f : (float)Q.lv[tid].val;
        if (tid == 0) {
            if (Q.fail) A.status[t] |= OGQ_ST_INTERNAL;
            st->done = 1;
        }
    }
    __syncthreads();
}

__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(kSolveThreads, 1) k_sel_round3(SelArgs A)
{
    Table& tb = sel_table();
    SolverShared& S = sel_state();
    __shared__ int sh_last;
    uint32_t* hist = sel_hist();
    pdl_wait();
    pdl_launch_dependents();
    const unsigned nitems = __ldcg(A.ws.nitems), ncells = __ldcg(A.ws.nitems + 1);
    for (unsigned w = blockIdx.x / kCluster; w < ncells; w += gridDim.x / kCluster)
        tensor_from_cells(A, __ldcg(&A.ws.items[(size_t)A.T * kMaxSlices - 1 - w].x), (int)(blockIdx.x % kCluster));

    for (unsigned w = blockIdx.x; w < nitems; w += gridDim.x) {
        const int2 it = A.ws.items[w];
        const int t = it.x;
        TState* st = A.ws.st + t;
        const int64_t tbeg = __ldg(A.off + t), tend = __ldg(A.off + t + 1);
        const unsigned ns = __ldcg(&st->expected);
        const bool from_grad = __ldcg(&st->from_grad) != 0;  // round 2's copies were cut short: slices of the tensor
        const int64_t cnt = from_grad ? tend - tbeg : (int64_t)__ldcg(&st->cursor[0]);
        int64_t per = (cnt + ns - 1) / ns;
        per = (per + 3) & ~(int64_t)3;
        int64_t pb_ = per * it.y, pe_ = pb_ + per;
        if (pb_ > cnt) pb_ = cnt;
        if (pe_ > cnt) pe_ = cnt;
        __syncthreads();
        table_from_intervals(tb, st->iv, __ldcg(&st->m));
        const bool copy_only = __ldcg(&st->compact_only) != 0;
        __syncthreads();
        if (!copy_only) zero_hist(hist, tb.ncells);
        __syncthreads();
        if (from_grad) {
            build_prefilter(tb, A.scheme == OGQ_BINGRAD_PB);
            grad_pass<kSolveThreads>(A, t, tbeg, tend, tbeg + pb_, tbeg + pe_, 1, copy_only);
        } else {
            Stager stg;
            stg.stage = sel_stage() + (threadIdx.x >> 5) * kStageCap;
            stg.dst = A.ws.buf[1] + sel_region(tbeg);
            stg.cursor = &st->cursor[1];
            stg.fill = 0;
            stream_piece(A.ws.buf[0], sel_region(tbeg) + pb_, sel_region(tbeg) + pe_, tb, hist, hist + kCells, hist + 2 * kCells, stg, copy_only);
            stg.flush();
        }
        __syncthreads();
        if (!copy_only) flush_hist(hist, tb.ncells, A.ws.gcnt + (size_t)t * kCells, A.ws.glsum + (size_t)t * kCells);
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned prev = atomicAdd(&st->arrive, 1u);
            sh_last = (prev == ns - 1);
        }
        __syncthreads();
        if (!sh_last) continue;
        __threadfence();
        if (copy_only) {
            finish_sorted(st, t, A.scheme == OGQ_BINGRAD_PB, A.s, A.ws.buf[1] + sel_region(tbeg), A.levels, A.status, 1);
            continue;
        }
        const int round = solver_load(st, S, A.scheme == OGQ_BINGRAD_PB, A.s);
        if (!solver_round(st, t, A.ws.gcnt + (size_t)t * kCells, A.ws.glsum + (size_t)t * kCells, A.scheme, A.s,
                          A.levels, A.status, A.ws.nitems, A.ws.items, A.ws.buf[1] + sel_region(tbeg), false, sel_region(tend) - sel_region(tbeg), round))
            finish_alone(A, t);
    }
}

cudaError_t launch_levels_select(const float* d_grad, const int64_t* d_off, int T, int64_t total, int scheme,
                                 int s, const float* d_tau, float* d_levels, int32_t* d_status, void* d_ws,
                                 size_t /*ws_bytes*/, int sm_count, cudaStream_t stream)
{
    {
        // the kernels need more dynamic shared memory than the default limit: raised once per device
        static std::atomic<bool> attr_set[64];
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= 64 || !attr_set[dev].load(std::memory_order_acquire)) {
            struct { void (*kernel)(SelArgs); size_t bytes; } limits[] = {{k_sel_round1, kStreamBytes}, {k_sel_round2, kStreamBytes},
                {k_sel_solve1, kSolve1Bytes}, {k_sel_solve2, kSolveBytes}, {k_sel_round3, kSolveBytes}};
            for (auto& l : limits) {
                e = cudaFuncSetAttribute(l.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)l.bytes);
                if (e != cudaSuccess) return e;
            }
            if (dev >= 0 && dev < 64) attr_set[dev].store(true, std::memory_order_release);
        }
    }
    // Flat streaming CTAs: one wave (kSelResident per SM).  Each CTA pays a set-up and a flush of its
    // cells per tensor piece, so larger shares stream more of the time.
    const int64_t wave = (int64_t)kSelResident * sm_count;
    const int target = wave < kMaxFlatCtas ? (int)wave : kMaxFlatCtas;
    FlatGrid g = make_flat_grid(total, target, T > kMaxShared ? 16384 : kMinShare);
    SelArgs A;
    A.grad = d_grad; A.tau = d_tau; A.off = d_off; A.T = T; A.total = total; A.chunk = T > kMaxShared ? g.chunk : 0;
    A.scheme = scheme; A.s = s; A.levels = d_levels; A.status = d_status;
    A.ws = sel_carve(d_ws, T, total);
    cudaError_t e = cudaSuccess;
    auto run = [&](const char* name, void (*kernel)(SelArgs), int ctas, size_t smem, int threads = kSelThreads) {
        if (e != cudaSuccess) return;
        launch_begin(name, stream);
        e = launch_pdl(kernel, ctas, threads, smem, stream, A);
        launch_end(stream);
    };
    A.first = total > kSmallN ? 0 : 1;
    const bool streams = total > kSmallN;  // some tensor may be larger than one CTA settles on its own
    if (streams) {
        run("k_sel_prepare", k_sel_prepare, T, 0);
        run("k_sel_round1", k_sel_round1, g.ctas, kStreamBytes);
        run("k_sel_solve1", k_sel_solve1, T, kSolve1Bytes, kSolveThreads);
        run("k_sel_round2", k_sel_round2, g.ctas, kStreamBytes);
    }
    run("k_sel_solve2", k_sel_solve2, T, kSolveBytes, kSolveThreads);
    if (streams) {
        // a cluster per tensor that may have that many candidates (its copies have room for an eighth of it); an empty launch of
        // eight clusters takes 2.9 us, of one 1.5
        const int64_t clusters = std::min<int64_t>(std::min<int64_t>(T, total / (kBufDiv * kSortN)), kMaxSlices / kCluster);
        run("k_sel_round3", k_sel_round3, (int)std::max<int64_t>(clusters, 1) * kCluster, kSolveBytes, kSolveThreads);
    }
    return e;
}

}  // namespace ogq

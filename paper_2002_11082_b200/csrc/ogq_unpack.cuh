// Pieces of the server step shared by the bucket-wide kernel and the fixed-length-bucket kernel: the levels of
// eight consecutive elements of one lane, summed over the workers in worker order.
//
// Level rows: one shared-memory read per element and worker from the worker's row of 2^BITS levels (free of bank
// conflicts, a row is at most 32 words).  1- and 2-bit codes have a table besides: the codes of the first eight
// (four) workers are transposed, in registers, into one index per element, and a table of 256 sums, built
// once per tensor in worker order, gives the sum of all of them in one read.
//   What bounds it: for the wider codes a shared-memory read and the instructions for its address per element and worker, and the
// wait for the words from L2, of which more in flight would not fit the registers (asked for a trip ahead in registers: 57
// instead of 52 us for the ResNet-50 bucket, eight workers of nine levels); for 1-bit codes DRAM.
#pragma once

#include <type_traits>

#include "ogq_common.cuh"
#include "ogq_quant.cuh"

namespace ogq {

template <int BITS>
constexpr int kTableWorkers = BITS == 1 ? 8 : BITS == 2 ? 4 : 0;  // workers that the table of sums takes in (0: no table)
template <int BITS>
constexpr int kTableFloats = kTableWorkers<BITS> ? 256 : 0;
// Workers whose words are loaded before any is used, and those of the last batch, which may be a full one.  That number is a template
// argument of the kernels: a kernel then has no condition between the reads of one worker's levels and the next's, which kept them from
// overlapping, and no instructions but its own (20 M elements of nine levels: two workers 26.9 -> 21 us, five 38 -> 32; 17 levels,
// seven 55 -> 45).  Eight at a time but for 3-bit codes, where four were as fast with half the instructions to fetch.
//   The last full batch outside the loop as well: in the loop its words are waited for batch by batch (VGG-19 bucket, a loop for all full
// batches and this: nine levels, eight workers 301 and 291 us; 17 levels, eight 370 and 351; 1-bit codes, twelve 277 and 242).
template <int BITS>
constexpr int kBatch = BITS == 1 || BITS == 3 ? 4 : 8;
// Workers of the last batch, at most.  Behind the table of 1-bit codes it is a double one, which takes in up to sixteen workers without a
// loop (VGG-19 bucket, sixteen: 403 us in the loop, 326 so).
template <int BITS, bool TABLE>
constexpr int kLast = TABLE && BITS == 1 ? 2 * kBatch<BITS> : kBatch<BITS>;
// In place of that number, 1-bit codes: the table of sums takes in all workers, up to eight (kTableOnly) or four of them.
constexpr int kTableOnly = -1;
template <int BITS, bool TABLE>
int rest_of(int K, bool quads = false)
{
    const int rows = K - (TABLE ? kTableWorkers<BITS> : 0);
    if (rows > kLast<BITS, TABLE>) return kLast<BITS, TABLE> - kBatch<BITS> + 1 + (rows - kLast<BITS, TABLE> - 1) % kBatch<BITS>;
    return rows > 0 ? rows : TABLE && BITS == 1 && quads ? (K > 4 ? kTableOnly : kTableOnly - 1) : 0;
}
template <int BITS>
constexpr int kRowStride = 1 << BITS;  // floats per level row: every code a field can hold has an entry

// The codes of eight elements of one worker as they lie in memory: bits [0, 8 BITS).
template <int BITS>
struct EightCodes {
    uint32_t lo, hi;  // hi: BITS = 5 only
};

// base: the first word of a group of 256 elements (8 BITS words), lane: which eight of them.
template <int BITS>
__device__ __forceinline__ EightCodes<BITS> load_codes(const uint32_t* __restrict__ base, int lane)
{
    EightCodes<BITS> c;
    c.hi = 0u;
    if constexpr (BITS == 1) {
        c.lo = __ldcg(reinterpret_cast<const unsigned char*>(base) + lane);
    } else if constexpr (BITS == 2) {
        c.lo = __ldcg(reinterpret_cast<const unsigned short*>(base) + lane);
    } else if constexpr (BITS == 4) {
        c.lo = __ldcg(base + lane);
    } else if constexpr (BITS == 3) {
        const int bit = 24 * lane, sh = bit & 31;
        const uint32_t* p = base + (bit >> 5);
        const uint32_t a = __ldcg(p), b = sh > 8 ? __ldcg(p + 1) : 0u;
        c.lo = __funnelshift_r(a, b, sh);
    } else {
        const int bit = 40 * lane, sh = bit & 31;
        const uint32_t* p = base + (bit >> 5);
        const uint32_t a = __ldcg(p), b = __ldcg(p + 1);
        c.lo = __funnelshift_r(a, b, sh);
        c.hi = b >> sh;
    }
    return c;
}

// launch(std::integral_constant<int, REST>) for the number of workers in the last batch.
template <int BITS, bool TABLE, int R = kLast<BITS, TABLE>, class Launch>
cudaError_t with_rest(int rest, Launch launch)
{
    if (rest == R) return launch(std::integral_constant<int, R>());
    if constexpr (R > (TABLE && BITS == 1 ? kTableOnly - 1 : TABLE && kTableWorkers<BITS> ? 0 : 1)) return with_rest<BITS, TABLE, R - 1>(rest, launch);
    else return cudaErrorInvalidValue;
}

// Shared addresses of the levels of the eight codes in the row at `row`, a multiple of the row's size (4-bit codes: of 256): it
// comes in with the instruction that isolates the code.
template <int BITS>
__device__ __forceinline__ void code_addresses(const EightCodes<BITS>& c, uint32_t row, uint32_t (&o)[8])
{
    if constexpr (BITS == 4) {
        const uint32_t even = (c.lo << 2) & 0x3c3c3c3cu, odd = (c.lo >> 2) & 0x3c3c3c3cu;  // one byte per code, times 4
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            o[2 * j] = __byte_perm(even, row, 0x7650 + j);
            o[2 * j + 1] = __byte_perm(odd, row, 0x7650 + j);
        }
    } else {
        constexpr uint32_t mask = ((1u << BITS) - 1u) << 2;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int b = j * BITS;
            uint32_t x;
            if (b < 2) x = c.lo << (2 - b);
            else if (b + BITS <= 32) x = c.lo >> (b - 2);
            else if (b < 32) x = __funnelshift_r(c.lo, c.hi, b - 2);
            else x = b - 32 < 2 ? c.hi << (2 - (b - 32)) : c.hi >> (b - 34);
            o[j] = (x & mask) | row;
        }
    }
}

template <int OFFSET>
__device__ __forceinline__ float load_level(uint32_t at)
{
    float x;
    asm("ld.shared.f32 %0, [%1+%2];" : "=f"(x) : "r"(at), "n"(OFFSET));
    return x;
}

// Two fp32 additions in one instruction (each rounded to nearest): (a0, a1) += (b0, b1).
__device__ __forceinline__ void add2(float& a0, float& a1, float b0, float b1)
{
    unsigned long long a, b;
    asm("mov.b64 %0, {%1, %2};" : "=l"(a) : "f"(a0), "f"(a1));
    asm("mov.b64 %0, {%1, %2};" : "=l"(b) : "f"(b0), "f"(b1));
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(a) : "l"(b));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a0), "=f"(a1) : "l"(a));
}

// acc += the levels of the codes of worker u of those whose rows begin at `row`.
template <int BITS, int U>
__device__ __forceinline__ void add_levels(const EightCodes<BITS>& c, uint32_t row, float (&acc)[8])
{
    uint32_t o[8];
    code_addresses<BITS>(c, row, o);
#pragma unroll
    for (int j = 0; j < 8; j += 2)
        add2(acc[j], acc[j + 1], load_level<U * kRowStride<BITS> * 4>(o[j]), load_level<U * kRowStride<BITS> * 4>(o[j + 1]));
}

// `words` and the sums of N workers whose rows begin at `row`: all words are loaded before any is used, and no condition comes
// between the workers (a branch after each kept the reads of one from overlapping those of the next).
template <int BITS, int G, int N, int U = 0>
__device__ __forceinline__ void add_batch(const EightCodes<BITS> (&c)[G][N], uint32_t row, float (&acc)[G][8])
{
    if constexpr (U < N) {
#pragma unroll
        for (int g = 0; g < G; ++g) add_levels<BITS, U>(c[g][U], row, acc[g]);
        add_batch<BITS, G, N, U + 1>(c, row, acc);
    }
}
template <int BITS, int G, int N, class Word>
__device__ __forceinline__ void sum_batch(int k0, int lane, uint32_t row, Word word, float (&acc)[G][8])
{
    EightCodes<BITS> c[G][N];
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
        for (int u = 0; u < N; ++u) c[g][u] = load_codes<BITS>(word(k0 + u, g), lane);
    add_batch<BITS, G, N>(c, row, acc);
}
// Table indices of eight elements from the codes of the kTableWorkers workers of a table (of workers that do not exist any
// code: the table's entries do not depend on it): byte e of x[0], byte e - 4 of x[1] is the index of element e, worker u's code in its bits
// [u BITS, (u + 1) BITS).
template <int BITS>
__device__ __forceinline__ void table_indices(const uint32_t (&c)[kTableWorkers<BITS>], uint32_t (&x)[2])
{
    if constexpr (BITS == 1) {
        // 8 x 8 bit transpose by three rounds of exchanges (Warren, Hacker's Delight, section 7-3)
        uint32_t lo = c[0] | c[1] << 8 | c[2] << 16 | c[3] << 24, hi = c[4] | c[5] << 8 | c[6] << 16 | c[7] << 24, t;
        t = (lo ^ (lo >> 7)) & 0x00aa00aau; lo ^= t ^ (t << 7);
        t = (hi ^ (hi >> 7)) & 0x00aa00aau; hi ^= t ^ (t << 7);
        t = (lo ^ (lo >> 14)) & 0x0000ccccu; lo ^= t ^ (t << 14);
        t = (hi ^ (hi >> 14)) & 0x0000ccccu; hi ^= t ^ (t << 14);
        t = (lo ^ (hi << 4)) & 0xf0f0f0f0u;
        x[0] = lo ^ t;
        x[1] = hi ^ (t >> 4);
    } else {
        // two 4 x 4 transposes of 2-bit fields
        const uint32_t p = c[0] | c[1] << 16, q = c[2] | c[3] << 16;
        x[0] = __byte_perm(p, q, 0x6420);
        x[1] = __byte_perm(p, q, 0x7531);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t z = x[h], t;
            t = (z ^ (z >> 6)) & 0x00cc00ccu; z ^= t ^ (t << 6);
            t = (z ^ (z >> 12)) & 0x0000f0f0u; z ^= t ^ (t << 12);
            x[h] = z;
        }
    }
}

// Entry i (0 ... 255) of the table for K workers: the sum of the levels that the codes in i stand for, in worker
// order.  level(k, code): level of worker k.
template <int BITS, class Level>
__device__ __forceinline__ float table_entry(int i, int K, Level level)
{
    float v[kTableWorkers<BITS>], a = 0.f;
#pragma unroll
    for (int u = 0; u < kTableWorkers<BITS>; ++u)
        v[u] = u < K ? level(u, (i >> (u * BITS)) & ((1 << BITS) - 1)) : 0.f;
#pragma unroll
    for (int u = 0; u < kTableWorkers<BITS>; ++u)
        if (u < K) a = __fadd_rn(a, v[u]);
    return a;
}

// The table's sums for eight elements; table: its shared address, a multiple of its size.
__device__ __forceinline__ void read_table(const uint32_t (&x)[2], uint32_t table, float (&acc)[8])
{
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const uint32_t w = x[j >> 2];
        const int b = 8 * (j & 3);
        acc[j] = load_level<0>(((b == 0 ? w << 2 : w >> (b - 2)) & 0x3fcu) | table);
    }
}

// Bytes of the level rows of K workers: rows begin at multiples of 256 bytes (see code_addresses).
template <int BITS>
__host__ __device__ constexpr uint32_t row_bytes(int K) { return ((uint32_t)K * kRowStride<BITS> * 4u + 255u) & ~255u; }

// Sums of the G groups of 256 elements at word(k, g) (worker k's first word of group g), eight elements of each for
// this lane.  table (not read unless TABLE), rows: shared addresses.  The words of several workers are loaded before any
// is used.
template <int BITS, int G, bool TABLE, int REST, class Word>
__device__ __forceinline__ void sum_workers(int K, int lane, uint32_t table, uint32_t rows, Word word, float (&acc)[G][8])
{
    constexpr int W = TABLE ? kTableWorkers<BITS> : 0, B = kBatch<BITS>;
    static_assert(BITS != 4 || B * kRowStride<BITS> * 4 % 256 == 0, "a batch's rows begin at a multiple of 256 bytes");
    int k0 = 0;
    if constexpr (W > 0) {
        uint32_t c[G][W], x[2];
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int u = 0; u < W; ++u) c[g][u] = u < K ? load_codes<BITS>(word(u, g), lane).lo : 0u;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            table_indices<BITS>(c[g], x);
            read_table(x, table, acc[g]);
        }
        k0 = W;
    } else {
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[g][j] = 0.f;
    }
    if constexpr (REST > 0)
        for (; k0 + kLast<BITS, TABLE> < K; k0 += B) sum_batch<BITS, G, B>(k0, lane, rows + (uint32_t)k0 * (kRowStride<BITS> * 4u), word, acc);
    if constexpr (REST > 0) sum_batch<BITS, G, REST>(k0, lane, rows + (uint32_t)k0 * (kRowStride<BITS> * 4u), word, acc);
}

// (WIDE: on a 32-byte boundary with one 256-bit store.  Two 128-bit stores write every 32-byte sector twice, half of it each time: 54.5
// -> 52.2 us for the ResNet-50 bucket at eight workers of nine levels, 32 -> 29.3 for 20 M elements of four workers of five.)
// Stores eight consecutive floats per lane at p (p: the lane's first, 32 bytes times lane above the warp's first),
// whose address is `shift` floats above a 16-byte boundary, with 128-bit stores: lanes pass their last
// `shift` values on to the next lane, the warp's two ends are stored one by one.
template <bool WIDE>
__device__ __forceinline__ void store8(float* p, int shift, int lane, const float (&v)[8])
{
    if (shift == 0) {
        if (WIDE && (reinterpret_cast<uintptr_t>(p) & 31) == 0) {  // (the same in all lanes)
            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" :: "l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]),
                         "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
            return;
        }
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<float4*>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
        return;
    }
    const float a = __shfl_up_sync(0xffffffffu, v[5], 1), b = __shfl_up_sync(0xffffffffu, v[6], 1),
                c = __shfl_up_sync(0xffffffffu, v[7], 1);
    float4 first, second;
    if (shift == 1) { first = make_float4(c, v[0], v[1], v[2]); second = make_float4(v[3], v[4], v[5], v[6]); }
    else if (shift == 2) { first = make_float4(b, c, v[0], v[1]); second = make_float4(v[2], v[3], v[4], v[5]); }
    else { first = make_float4(a, b, c, v[0]); second = make_float4(v[1], v[2], v[3], v[4]); }
    if (lane > 0) {
        *reinterpret_cast<float4*>(p - shift) = first;
    } else {
        p[0] = v[0];
        if (shift < 3) p[1] = v[1];
        if (shift < 2) p[2] = v[2];
    }
    *reinterpret_cast<float4*>(p - shift + 4) = second;
    if (lane == 31) {
        p[7] = v[7];
        if (shift > 1) p[6] = v[6];
        if (shift > 2) p[5] = v[5];
    }
}

}  // namespace ogq

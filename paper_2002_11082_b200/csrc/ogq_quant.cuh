// Per-element pieces of the quantizer shared by the bucket-wide kernel and the fixed-length-bucket
// kernel: segment search in a shared-memory level table, the rounding decision, word assembly.
#pragma once

#include "ogq_common.cuh"

namespace ogq {

constexpr int kMaxLevels = 32;
constexpr int kMaxWorkers = 64;

// Combines the 4*BITS-bit chunk of each lane into the 4*BITS words of a 128-element group.  A word whose
// width is a whole number of chunks (BITS = 1, 2, 4) is OR-ed together by a butterfly inside its 8, 4 or
// 2 lanes.  3- and 5-bit chunks straddle words: eight lanes hold 3 or 5 words, and lane i of the eight
// fetches the three or four chunks that touch word i by shuffle and puts them into place.  Registers only: OR-ing the chunks
// together with shared-memory atomics serialised on the words that neighbouring lanes share.
// The lanes with packs_word() true then hold word packed_word() of the group.
template <int BITS>
__device__ __forceinline__ bool packs_word(int lane)
{
    constexpr bool kPow2 = (BITS & (BITS - 1)) == 0;
    constexpr int L = kPow2 ? 8 / BITS : 1;
    return kPow2 ? (lane & (L - 1)) == 0 : (lane & 7) < BITS;
}

template <int BITS>
__device__ __forceinline__ int packed_word(int lane)
{
    constexpr bool kPow2 = (BITS & (BITS - 1)) == 0;
    constexpr int L = kPow2 ? 8 / BITS : 1;
    return kPow2 ? lane / L : (lane >> 3) * BITS + (lane & 7);
}

template <int BITS>
__device__ __forceinline__ uint32_t assemble_words(uint32_t chunk, int lane)
{
    if constexpr ((BITS & (BITS - 1)) == 0) {
        constexpr int L = 8 / BITS;
        uint32_t x = chunk << (4 * BITS * (lane & (L - 1)));
#pragma unroll
        for (int o = 1; o < L; o <<= 1) x |= __shfl_xor_sync(0xffffffffu, x, o);
        return x;
    } else {
        constexpr int W = 4 * BITS;                 // bits per lane
        const int bit = (lane & 7) * 32;            // first bit of this lane's word inside the eight chunks
        const int a = (lane & 24) + bit / W, o = bit % W;
        uint32_t x = __shfl_sync(0xffffffffu, chunk, a) >> o;
        // (shifted into place by a multiplication with 2^shift, or with 0 for a chunk past the word: a multiply-add
        // in place of a shift and an OR, on the less busy pipe)
#pragma unroll
        for (int u = 1; u <= (BITS == 3 ? 3 : 2); ++u) {
            const uint32_t scale = u * W - o < 32 ? 1u << (u * W - o) : 0u;
            x += __shfl_sync(0xffffffffu, chunk, (a + u) & 31) * scale;
        }
        return x;
    }
}

// The quantizer's table of one tensor or bucket in shared memory: entry k = {level k, width of the segment
// above it, times 2^-24}.  The rounding decision u w < d 2^24 (u: 24 random bits, w: width, d: distance to
// the lower level, every operation rounded to fp32) is taken as u (w 2^-24) < d, which is the same decision
// as long as scaling by 2^24 neither overflows nor leaves the normal numbers: quant_table_scales() tells,
// for the whole table; other tables go through the slow path, which does the operations as written.
__device__ __forceinline__ float2 quant_table_entry(float level, float next)
{
    return make_float2(level, __fmul_rn(__fsub_rn(next, level), 0x1p-24f));
}
__device__ __forceinline__ bool quant_table_scales(float level, float next)
{
    const float w = __fsub_rn(next, level);
    return fabsf(level) < 0x1p100f && fabsf(next) < 0x1p100f && (w == 0.f || w >= 0x1p-100f);
}

// Byte distances in the table, as kernel parameters: {8, 16, 32} are one, two and four entries.
struct QuantSteps {
    uint32_t one, b8, b16, b32;
};
inline QuantSteps quant_steps() { return QuantSteps{1u, 8u, 16u, 32u}; }

// Segment search and rounding decision of one element.  `tab` is the shared address of the table, `mid` its
// middle level.  Returns the address of the entry whose index is the element's
// code: the entry of the segment's lower level, or the next one when the element rounds up.
//   28 instructions per element at s = 9, ten of them Philox.  What bounds the quantizer are the pipes these share, not its loads:
// pinned to one block in the cache it takes 183 us for 143.7 M elements, with its own loads 191, without Philox 130.  A wide
// multiplication holds the multiply pipe for four cycles and the integer pipe for two, a comparison or logic instruction the integer
// pipe for two: 36 cycles of the integer pipe per 32 elements, 28 of the other, 49 measured.  So the conditional steps are multiply-adds, which go to the
// other pipe; both factors are parameters (1 and the distance), a plain addition or a known power of two
// would become an integer-pipe instruction.
template <int STEP>
__device__ __forceinline__ void search_step(uint32_t& a, float v, const QuantSteps& st)
{
    asm("{ .reg .pred p; .reg .f32 t; ld.shared.f32 t, [%0+%2]; setp.le.f32 p, t, %1; @p mad.lo.u32 %0, %3, %4, %0; }"
        : "+r"(a) : "f"(v), "n"(STEP * 8), "r"(st.one), "r"(STEP == 1 ? st.b8 : STEP == 2 ? st.b16 : st.b32));
}

template <int BITS>
__device__ __forceinline__ uint32_t entry_after_rounding(float v, uint32_t rnd, uint32_t tab, float mid, const QuantSteps& st)
{
    uint32_t a = tab;
    if constexpr (BITS >= 2) {
        a = (mid <= v) ? tab + (8u << (BITS - 2)) : tab;
        if constexpr (BITS >= 5) search_step<4>(a, v, st);
        if constexpr (BITS >= 4) search_step<2>(a, v, st);
        if constexpr (BITS >= 3) search_step<1>(a, v, st);
    }
    float lo, w;
    if constexpr (BITS == 1) {  // the only entry: a load that the compiler may move, but not past a barrier
        const float2 e = *static_cast<const float2*>(__cvta_shared_to_generic(tab));
        lo = e.x; w = e.y;
    } else {
        asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(lo), "=f"(w) : "r"(a));
    }
    const float lhs = __fmul_rn((float)(rnd >> 8), w);
    const float rhs = __fsub_rn(v, lo);
    asm("{ .reg .pred p; setp.lt.f32 p, %1, %2; @p mad.lo.u32 %0, %3, %4, %0; }"
        : "+r"(a) : "f"(lhs), "f"(rhs), "r"(st.one), "r"(st.b8));
    return a;
}

// The same for tables that do not scale, with the operations as written: level(k) returns level k.
template <int BITS, class Level>
__device__ __forceinline__ uint32_t code_as_written(float v, uint32_t rnd, Level level)
{
    int k = 0;
#pragma unroll
    for (int step = (BITS >= 2) ? (1 << (BITS - 2)) : 0; step >= 1; step >>= 1)
        if (level(k + step) <= v) k += step;
    const float lo = level(k);
    const float lhs = __fmul_rn((float)(rnd >> 8), __fsub_rn(level(k + 1), lo));
    const float rhs = __fmul_rn(__fsub_rn(v, lo), 16777216.0f);
    return (uint32_t)k + ((lhs < rhs) ? 1u : 0u);
}

// The codes of four elements from their entries' addresses (entries are 8 bytes apart): BITS bits each, the
// first element lowest.
template <int BITS>
__device__ __forceinline__ uint32_t codes_of_entries(uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t tab)
{
    // the sum carries this multiple of the table's address
    const uint32_t base = tab * (1u + (1u << BITS) + (1u << (2 * BITS)) + (1u << (3 * BITS)));
    return (a0 + (a1 << BITS) + (a2 << (2 * BITS)) + (a3 << (3 * BITS)) - base) >> 3;
}

// Stores the 4*BITS-bit chunks of a warp's 128 elements at `out` (4*BITS words), as bytes or half-words: lanes whose
// chunks are whole bytes on their own, the others after one exchange with their neighbour (a pair's 4-bit chunks make
// one byte, its 12-bit chunks three, its 20-bit chunks five).  L2 puts the bytes together; building words of
// 12- and 20-bit chunks first took up to four shuffles.
template <int BITS>
__device__ __forceinline__ void store_chunks(uint32_t* out, uint32_t chunk, int lane)
{
    if constexpr (BITS == 4) {
        reinterpret_cast<uint16_t*>(out)[lane] = (uint16_t)chunk;
    } else if constexpr (BITS == 2) {
        reinterpret_cast<uint8_t*>(out)[lane] = (uint8_t)chunk;
    } else {
        const uint32_t other = __shfl_xor_sync(0xffffffffu, chunk, 1);
        const bool even = (lane & 1) == 0;
        if constexpr (BITS == 1) {
            if (even) reinterpret_cast<uint8_t*>(out)[lane >> 1] = (uint8_t)(chunk | other << 4);
        } else {
            constexpr int kEven = (BITS + 1) / 2;  // bytes of the even lane; the odd lane stores the others
            uint8_t* p = reinterpret_cast<uint8_t*>(out) + BITS * (lane >> 1) + (even ? 0 : kEven);
            const uint32_t v = even ? chunk | other << (4 * BITS) : chunk >> 4;
            p[0] = (uint8_t)v;
            if (BITS == 5) p[1] = (uint8_t)(v >> 8);
            if (even) p[BITS / 2] = (uint8_t)(v >> (8 * (BITS / 2)));
        }
    }
}

}  // namespace ogq

// Nested codes from their 2-bit fields, whole words at a time.
//
// A word of a 2-bit field holds four k32 steps on top of each other (fq_layout.cuh), at the same bit offsets in every field.  So
// two fields become 4-bit codes with one three-input select per word (even steps in one word, odd steps in the other), and two
// such words become bytes with one more: about three operations per step and four codes for all eight bits, against a shift and an
// AND-OR per field when each step is taken out of each field by itself.
#pragma once
#include <cstdint>

#include "fq_layout.cuh"

namespace fq {

// Bits of a where MASK is set, of b elsewhere: one LOP3.
template <uint32_t MASK>
__device__ __forceinline__ uint32_t pick(uint32_t a, uint32_t b) { return (a & MASK) | (b & ~MASK); }

// 4-bit codes of two fields: steps 0 (low nibbles) and 2 (high nibbles) in `even`, 1 and 3 in `odd`.
__device__ __forceinline__ void merge_nibbles(uint32_t upper, uint32_t lower, uint32_t& even, uint32_t& odd)
{
    even = pick<0xccccccccu>(upper << 2, lower);
    odd = pick<0xccccccccu>(upper, lower >> 2);
}

// The words of the first N fields, two or more -> the parent's bytes of steps 0 .. 3, dropped bits zero (of the last field the upper KEEP bits count).
template <int N, int KEEP>
__device__ __forceinline__ void merge_bytes(const uint32_t (&w)[4], uint32_t (&step)[4])
{
    constexpr uint32_t kPair = 0xccccccccu, kHigh = 0xf0f0f0f0u;
    static_assert(N >= 2 && N <= 4 && (KEEP == 1 || KEEP == 2), "fields of a nested child");
    uint32_t ue, uo;
    merge_nibbles(w[0], w[1], ue, uo);
    if constexpr (N == 2) {
        constexpr uint32_t m = KEEP == 2 ? kHigh : 0xe0e0e0e0u;
        step[0] = (ue << 4) & m; step[1] = (uo << 4) & m; step[2] = ue & m; step[3] = uo & m;
    } else {
        uint32_t ve, vo;
        if constexpr (N == 3) {
            constexpr uint32_t m = KEEP == 2 ? kPair : 0x88888888u;
            ve = (w[2] << 2) & m; vo = w[2] & m;
        } else {
            merge_nibbles(w[2], KEEP == 2 ? w[3] : w[3] & 0xaaaaaaaau, ve, vo);
        }
        step[0] = pick<kHigh>(ue << 4, ve); step[2] = pick<kHigh>(ue, ve >> 4);
        step[1] = pick<kHigh>(uo << 4, vo); step[3] = pick<kHigh>(uo, vo >> 4);
    }
}

}  // namespace fq

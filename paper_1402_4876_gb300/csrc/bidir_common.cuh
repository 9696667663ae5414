// What the seed sweep and the bidirectional kernel share: the pieces of a
// pattern and the rule for checking rows against the text.
#pragma once

#include "search_common.cuh"

namespace mica {

constexpr uint32_t SCHEME_FREE = 7;         // the single scheme of reads shorter than k + 1
constexpr uint32_t BD_VERIFY_MIN = 12;      // matched bases of a one-row node before it is checked against the text
constexpr uint32_t BD_VERIFY_LEFT = 8;      // ... when at least this many bases are left to match

// piece boundaries of a pattern of m bases in p pieces
// (i m <= 4 * 256, so the division by 3 is a multiplication: 21846 / 2^16 exceeds
// 1 / 3 by less than 2^-16, too little to carry 1024 / 3 past the next integer)
__device__ __forceinline__ uint32_t bnd(uint32_t i, uint32_t m, uint32_t p)
{
    const uint32_t x = i * m;
    return p == 3 ? (x * 21846u) >> 16 : x >> (p >> 1);
}

// The boundaries bnd(0) .. bnd(4) of a task's pieces as 9-bit fields (fields
// past p hold 511), computed once per task so that a node's scheme check
// needs no division.
__device__ __forceinline__ unsigned long long pack_bounds(uint32_t m, uint32_t p)
{
    unsigned long long v = 0;
#pragma unroll
    for (uint32_t i = 0; i <= 4; i++) v |= (unsigned long long)(i <= p ? bnd(i, m, p) : 511u) << (9 * i);
    return v;
}
__device__ __forceinline__ uint32_t bound_at(unsigned long long v, uint32_t i) { return (uint32_t)(v >> (9 * i)) & 511u; }
// the piece holding position pos: the boundaries 1..3 at or below it
__device__ __forceinline__ uint32_t piece_at(unsigned long long v, uint32_t pos)
{
    return (pos >= bound_at(v, 1)) + (pos >= bound_at(v, 2)) + (pos >= bound_at(v, 3));
}

}  // namespace mica

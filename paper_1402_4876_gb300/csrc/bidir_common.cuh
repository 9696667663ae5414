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

// node meta: slot (6 bits) | a (9) | b (9) | d (2) | d0 (2) | scheme (3)
__device__ __forceinline__ uint32_t bd_meta(uint32_t slot, uint32_t a, uint32_t b, uint32_t d, uint32_t d0,
                                            uint32_t j)
{
    return slot | (a << 6) | (b << 15) | (d << 24) | (d0 << 26) | (j << 28);
}
constexpr uint32_t BM_SLOT_MASK = 63u;
__device__ __forceinline__ uint32_t bm_slot(uint32_t x) { return x & BM_SLOT_MASK; }
__device__ __forceinline__ uint32_t bm_a(uint32_t x) { return (x >> 6) & 511u; }
__device__ __forceinline__ uint32_t bm_b(uint32_t x) { return (x >> 15) & 511u; }
__device__ __forceinline__ uint32_t bm_d(uint32_t x) { return (x >> 24) & 3u; }
__device__ __forceinline__ uint32_t bm_d0(uint32_t x) { return (x >> 26) & 3u; }
__device__ __forceinline__ uint32_t bm_j(uint32_t x) { return (x >> 28) & 7u; }

// May a child that extends P[a, b) by base c at position pos (to the left
// when a > 0, else to the right) exist under scheme j?  Returns the child's
// d0 (mismatches before its current left piece) through d0n.
__device__ __forceinline__ bool bd_allowed(uint32_t j, uint32_t a, uint32_t pos, unsigned long long bounds,
                                           uint32_t k, uint32_t d, uint32_t d0, uint32_t cost, uint32_t &d0n)
{
    const uint32_t dn = d + cost;
    d0n = d0;
    if (dn > k) return false;
    if (j == SCHEME_FREE || a == 0) return true;              // free scheme, or the right phase
    const uint32_t i = piece_at(bounds, pos);
    if (i == j) return cost == 0;                             // the exact piece
    // a piece left of j: it needs a substitution, and so do pieces 0 .. i - 1
    d0n = (a == bound_at(bounds, i + 1)) ? d : d0;            // entering piece i
    const uint32_t dp = dn - d0n;
    if (pos == bound_at(bounds, i)) return dp >= 1 && dn + i <= k;   // piece i complete
    return dn + i + (dp == 0 ? 1u : 0u) <= k;
}

// The last CTA of a launch: the nodes it put in the frontier become the next
// round's tasks.
__device__ __forceinline__ void end_round(SearchCtl *ctl, uint32_t cap)
{
    const uint32_t n = *(volatile unsigned *)&ctl->fr_count;
    ctl->spills += n;
    ctl->ntasks = min(n, cap);
    ctl->unfinished = (n ? 1u : 0u) | (*(volatile unsigned *)&ctl->redo_reads ? 2u : 0u) |
                      (*(volatile unsigned *)&ctl->pool_tasks ? 4u : 0u);
    ctl->rounds_run += n != 0;
    ctl->task_head = 0;
    ctl->fr_count = 0;
    ctl->done_ctas = 0;
}

}  // namespace mica

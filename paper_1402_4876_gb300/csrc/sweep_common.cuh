// What the sweep, the trees' kernel and the row checks share.
#pragma once

#include "bidir_common.cuh"

namespace mica {

// Rows of a tree's interval that is checked row by row: while bases are left to
// match on its left, which the rows' contexts are compared with, and after.
// Each tree ends sooner the larger they are, each check is more work: search
// kernels with 64, 16 / 128, 32 / 256, 64 / 400, 128 rows (in every launch, an item a
// warp): 512 Mbp human-like 1M
// mates 3.57 / 3.22 / 3.27 / 3.14 ms, 250 bp k = 3 0.54 / 0.51 / 0.45 / 0.47 ms,
// uneven 1M reads 1.39 / 1.46 / 1.54 / 1.55 ms.
constexpr uint32_t TREE_SPLIT_LEFT = 256;
constexpr uint32_t TREE_SPLIT_RIGHT = 64;
// ... above this many, in a launch whose lanes are all at work, only once an
// eighth of the rows that the lane began with have dropped out: copies that do
// not differ stay one interval to the end, where rows told apart are a leaf
// each.  A launch of fewer nodes takes as long as its longest chain, which row
// checks end.  100k reads of 100 bp inside 200 exact copies, cap 10 / cap 1000:
// 2.52 / 2.59 -> 1.08 / 1.19 ms; uneven 1M reads 2.03 -> 1.79.  With the rule in
// every launch the best of 100k x 250 bp took 0.97 ms instead of 0.87.
constexpr uint32_t TREE_SPLIT_FEW = 64;

// An item of rows to check is (row l, task, this word, the read's context): up
// to 511 rows, scheme j, context bases in the exact piece, budget k, pattern
// position of the matched bases, mismatches left to the bases around them.
__device__ __forceinline__ uint32_t item_meta(uint32_t rows, uint32_t j, uint32_t ex, uint32_t k, uint32_t at,
                                              uint32_t rem)
{
    return rows | (j << 9) | (ex << 11) | (k << 16) | (at << 18) | (rem << 27);
}

// Raw word i of a read, 0 outside it.
__device__ __forceinline__ uint32_t raw_word(const uint32_t *w, int i, int wn)
{
    return (i >= 0 && i < wn) ? __ldg(w + i) : 0u;
}

// The 16 bases of the pattern (the read, or its other strand) before position
// at, the nearest in the top bits, as the index keeps a row's; zeros past the
// pattern's start.
__device__ __forceinline__ uint32_t read_context(const uint32_t *w, uint32_t minus, uint32_t m, uint32_t at)
{
    const int wn = (int)((m + 15) >> 4);
    if (minus) {   // R[m - at, m - at + 16) complemented, back to front
        const uint32_t p = m - at;
        const int i = (int)(p >> 4);
        return rev_groups(~__funnelshift_r(raw_word(w, i, wn), raw_word(w, i + 1, wn), 2u * (p & 15u)));
    }
    if (at >= 16u) {
        const uint32_t p = at - 16u;
        const int i = (int)(p >> 4);
        return __funnelshift_r(raw_word(w, i, wn), raw_word(w, i + 1, wn), 2u * (p & 15u));
    }
    return at ? __ldg(w) << (2u * (16u - at)) : 0u;
}

// sweep.cu and tree.cu, for the host code of bidir.cu
int enqueue_sweep(const mica_index *idx, Workspace &w, const ReadsView &rd, uint32_t verify_min, uint32_t budget,
                  uint2 *list, uint4 *nodes, uint32_t *node_meta, uint32_t cap, uint4 *items, uint32_t item_cap,
                  cudaStream_t s, uint64_t &launches);
int enqueue_rows(const mica_index *idx, Workspace &w, const ReadsView &rd, uint4 *items, uint32_t item_cap,
                 cudaStream_t s, uint64_t &launches);
int launch_tree(const OccSide &fwd, const OccSide &rev, Workspace &w, const ReadsView &rd, uint32_t round,
                const uint4 *in, const uint32_t *in_meta, uint32_t in_cap, uint4 *out, uint32_t *out_meta, uint32_t cap,
                uint4 *items, uint32_t item_cap, uint32_t *redo, uint32_t verify_min, uint32_t tail, cudaStream_t s);
// What the trees' warps may still add to a list once it is found full: the
// nodes (items) each has staged, and those its lanes are at.
constexpr uint32_t TREE_WARPS = 152u * 3u * 8u;
constexpr uint32_t TREE_LAST = TREE_WARPS * 160u;

}  // namespace mica

// The seed sweep: the first pass of the bidirectional search (bidir.cu) when
// the whole suffix array and the text are resident.
//
// Most schemes of most reads need no search tree: the exact piece's last q
// bases come up empty in the seed table (a read's other strand, mostly) or
// name a few rows, each of which one look at the text decides.  The sweep does
// exactly those: one thread per (read, strand) looks its k + 1 seeds up, the
// rows of the small intervals are checked against the text 32 at a time, and
// only the schemes it cannot finish (an interval of many rows, a piece too
// short to be told apart, a read shorter than k + 1 bases) go on a task list
// with a bit per scheme, which the bidirectional kernel works through.
//
// What bounds it: random 32-byte reads of HBM (a table entry pair per seed, a
// suffix array entry per row; the text of a genome of this size is L2 hits), so
// it holds nothing but two short queues per warp and runs as many warps as the
// registers allow, to have as many of those reads in flight as there can be.
// The bidirectional kernel did the same lookups from 18 to 24 warps per SM
// with task slots, staged patterns and stacks around them, and read the
// reversed genome's table too, which only a tree's second interval needs.
//
// Measured on one GB300, search kernels of 1M x 150 bp reads, k = 2, on a 64
// Mbp genome with repeats: 1.57 ms before, 0.45 ms of sweep + 0.55 ms of trees
// with it (6M seeds and 2.4M windows at 30 G random reads/s would take 0.3 ms).
#include <algorithm>

#include "bidir_common.cuh"

namespace mica {
namespace {

constexpr unsigned SFULL = 0xffffffffu;
constexpr int SWEEP_WARPS = 8;
constexpr int SWEEP_CTAS = 4;     // per SM
constexpr uint32_t ROW_ITEM = 128;   // rows of an item (32 .. 256 within 2%)
constexpr int SWEEP_QUEUE = 64;   // intervals waiting: fewer than 32 left over (each has a row) plus 32 new ones

struct SweepArgs {
    QmerView seed;               // the longer table of G$ when there is one
    const uint2 *sa_ctx;
    const uint32_t *text;
    uint64_t n;
    ReadsView rd;
    SearchCtl *ctl;
    Interval *iv;
    uint32_t *iv_cnt;
    uint2 *list;                 // (task, schemes left as bits)
    // larger intervals, a piece of up to ROW_ITEM rows each: (row l, task, rows | scheme << 9 | context bases in
    // the exact piece << 11 | budget << 16 | pattern position of the matched bases << 18, the read's context)
    uint4 *items;
    uint32_t item_cap;
    uint32_t verify_min, split, split_max;
};

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

// One leaf per lane (where leaf): its interval, with one counter update per warp.
__device__ __forceinline__ void sweep_emit(const SweepArgs &a, bool leaf, uint32_t rid, uint32_t meta, uint32_t l,
                                           uint32_t r, int lane)
{
    const unsigned bal = __ballot_sync(SFULL, leaf);
    if (!bal) return;
    uint32_t at = 0;
    if (lane == 0) at = atomicAdd(&a.ctl->iv_count, (unsigned)__popc(bal));
    at = __shfl_sync(SFULL, at, 0) + __popc(bal & ((1u << lane) - 1u));
    if (leaf) {
        atomicAdd(&a.iv_cnt[rid], 1u);
        if (at < a.ctl->iv_cap) {
            Interval x;
            x.read = rid; x.meta = meta; x.l = l; x.r = r;
            a.iv[at] = x;
        } else {
            atomicOr(&a.ctl->error, ERR_IV_OVERFLOW);
        }
    }
}

// Does the window of m bases at text position s hold a placement of the read
// (words w, its other strand if minus) whose leftmost exact piece is piece j,
// with at most k mismatches?  At most k + 1 mismatches are looked at, each
// marking its piece: the scheme asks that no bit of piece j and every bit
// below it be set.  d: the mismatches; words: the text words read.
__device__ __forceinline__ bool sweep_check(const uint32_t *__restrict__ text, const uint32_t *__restrict__ w,
                                            uint32_t minus, uint32_t m, uint32_t k, uint32_t j, uint32_t s,
                                            uint32_t &d, uint32_t &words)
{
    const uint32_t p = k + 1;
    const uint32_t b1 = bnd(1, m, p), b2 = p >= 2 ? bnd(2, m, p) : 511u, b3 = p >= 3 ? bnd(3, m, p) : 511u;
    const uint32_t *tp = text + (s >> 4);
    const uint32_t sh = 2u * (s & 15u);
    const int wn = (int)((m + 15) >> 4);
    uint32_t tot = 0, hit = 0;
    uint32_t prev = __ldg(tp);
    words = 1;
    for (int q0 = 0; q0 < wn; q0 += 4) {
        uint32_t tw[4], rw[5];
#pragma unroll
        for (int i = 0; i < 4; i++) tw[i] = q0 + i < wn ? __ldg(tp + q0 + i + 1) : 0u;
#pragma unroll
        for (int i = 0; i < 5; i++) rw[i] = raw_word(w, minus ? wn - 1 - q0 - i : q0 + i, wn);
        words += (uint32_t)min(4, wn - q0);
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int q = q0 + i;
            const uint32_t pat = minus ? rc_word(rw[i], rw[i + 1], m) : rw[i];
            uint32_t x = pat ^ __funnelshift_r(prev, tw[i], sh);
            prev = tw[i];
            x = (x | (x >> 1)) & 0x55555555u & low_mask(2u * (uint32_t)min(max((int)m - 16 * q, 0), 16));
            while (x && tot <= k) {
                const uint32_t pos = 16u * (uint32_t)q + (uint32_t)(__ffs(x) - 1) / 2u;
                x &= x - 1;
                tot++;
                hit |= 1u << ((pos >= b1) + (pos >= b2) + (pos >= b3));
            }
        }
        if (tot > k || ((hit >> j) & 1u)) return false;
    }
    d = tot;
    return (hit & ((1u << j) - 1u)) == (1u << j) - 1u;
}

// A warp's queues: intervals whose rows are to be told apart by their left
// contexts, and the windows of the rows that pass, to be checked against the
// text.  Each holds fewer than 32 rows (windows) when a batch of 32 is added.
struct SweepQueue {
    // (row l, task, rows | scheme << 16 | context bases in the exact piece << 18 | budget << 23, the read's context)
    uint4 iv[SWEEP_QUEUE];
    uint16_t at[SWEEP_QUEUE];                             // pattern position of the interval's matched bases
    uint32_t start[SWEEP_QUEUE], task[SWEEP_QUEUE];       // windows: text position, task,
    uint8_t scheme[SWEEP_QUEUE];                          //   scheme
};

// 32 windows (or all that wait) against the text.
__device__ __forceinline__ void sweep_windows(const SweepArgs &a, const SweepQueue &Q, uint32_t &windows, int lane,
                                              uint32_t &c_verify, uint32_t &c_vbytes, uint32_t &c_vsect)
{
    const uint32_t take = min(windows, 32u);
    const uint32_t e = windows - 1u - (uint32_t)lane;
    windows -= take;
    bool leaf = false;
    uint32_t d = 0, s = 0, rid = 0, minus = 0;
    if ((uint32_t)lane < take) {
        s = Q.start[e];
        rid = Q.task[e] >> 1;
        minus = Q.task[e] & 1u;
        const uint32_t m = a.rd.len[rid], k = a.rd.k[rid];
        uint32_t words = 0;
        leaf = sweep_check(a.text, a.rd.words + a.rd.word_off[rid], minus, m, k, Q.scheme[e], s, d, words);
        c_verify++;
        c_vbytes += 4u * words;
        c_vsect += (((s >> 4) & 7u) * 4u + 4u * words + 31u) / 32u;
    }
    sweep_emit(a, leaf, rid, d | (minus << 2) | IV_POS, s, s + 1u, lane);
    __syncwarp();
}

// The rows of the newest intervals, 32 rows (or all that wait): a row stays
// when the bases before it differ from the read's nowhere in the exact piece
// and in at most its budget of the rest (they are only a part of what the
// text check looks at, so no placement is lost), and its window lies in G.
__device__ __forceinline__ void sweep_rows(const SweepArgs &a, SweepQueue &Q, uint32_t &top, uint32_t &rows,
                                           uint32_t &windows, int lane, uint32_t &c_vbytes, uint32_t &c_vsect)
{
    const uint32_t n = min(top, 32u);
    const uint32_t e = top - 1u - (uint32_t)lane;
    uint4 it = make_uint4(0, 0, 0, 0);
    uint32_t iat = 0;
    if ((uint32_t)lane < n) { it = Q.iv[e]; iat = Q.at[e]; }
    const uint32_t sz = it.z & 0xffffu;
    uint32_t incl = sz;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(SFULL, incl, o);
        if (lane >= o) incl += y;
    }
    const uint32_t excl = incl - sz;
    // row `lane` of the batch belongs to the last entry whose first row is not past it
    const unsigned heads = __reduce_or_sync(SFULL, (sz && excl < 32u) ? 1u << excl : 0u);
    const int src = __popc(heads & (0xffffffffu >> (31 - lane))) - 1;
    const uint32_t take = min(rows, 32u);
    const uint32_t first = __shfl_sync(SFULL, excl, src);
    const uint32_t row = __shfl_sync(SFULL, it.x, src) + ((uint32_t)lane - first);
    const uint32_t task = __shfl_sync(SFULL, it.y, src), meta = __shfl_sync(SFULL, it.z, src);
    const uint32_t ctx = __shfl_sync(SFULL, it.w, src), at = __shfl_sync(SFULL, iat, src);
    const uint32_t gone = __popc(__ballot_sync(SFULL, sz && incl <= 32u));
    if (sz && excl < 32u && incl > 32u) {   // the rest of a partly taken interval stays on top
        Q.iv[e].x = it.x + (32u - excl);
        Q.iv[e].z = it.z - (32u - excl);
    }
    top -= gone;
    rows -= take;
    bool stay = false;
    uint32_t s = 0;
    if ((uint32_t)lane < take) {
        const uint2 x = __ldg(a.sa_ctx + row);
        const uint32_t m = a.rd.len[task >> 1];
        s = x.x - at;
        uint32_t df = x.y ^ ctx;
        df = (df | (df >> 1)) & 0x55555555u;
        if (at < 16u) df &= at ? ~0u << (2u * (16u - at)) : 0u;          // context bases the pattern has
        const uint32_t ex = (meta >> 18) & 31u;                          // ... and those in the exact piece
        const bool exact = ex == 0 || (df >> (2u * (16u - ex))) == 0;
        stay = x.x >= at && (uint64_t)s + m <= a.n && exact && __popc(df) <= ((meta >> 23) & 3u);
        c_vbytes += 8u;
        if (lane == 0 || (row & 3u) == 0 || first == (uint32_t)lane) c_vsect++;
    }
    const unsigned bal = __ballot_sync(SFULL, stay);
    if (stay) {
        const uint32_t q = windows + __popc(bal & ((1u << lane) - 1u));
        Q.start[q] = s;
        Q.task[q] = task;
        Q.scheme[q] = (uint8_t)((meta >> 16) & 3u);
    }
    windows += __popc(bal);
    __syncwarp();
}

// Put the warp's intervals of many rows (lanes with `want`) on the item list,
// with one counter update; false for a lane whose items do not fit (what was
// reserved for them is filled with empty items).
__device__ __forceinline__ bool sweep_items(const SweepArgs &a, bool want, uint32_t l, uint32_t sz, uint32_t task,
                                            const uint32_t *w, uint32_t m, uint32_t k, uint32_t j, uint32_t qe,
                                            int lane)
{
    if (!__any_sync(SFULL, want)) return false;
    const uint32_t n = want ? (sz + ROW_ITEM - 1) / ROW_ITEM : 0u;
    uint32_t incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(SFULL, incl, o);
        if (lane >= o) incl += y;
    }
    uint32_t q = 0;
    if (lane == 31) q = atomicAdd(&a.ctl->row_items, incl);
    q = __shfl_sync(SFULL, q, 31) + incl - n;
    if (!want || q >= a.item_cap) return false;
    const bool fits = n <= a.item_cap - q;
    const uint32_t at = bnd(j + 1, m, k + 1) - qe;
    const uint32_t meta = (j << 9) | (min(16u, at - bnd(j, m, k + 1)) << 11) | (k << 16) | (at << 18);
    const uint32_t ctx = read_context(w, task & 1u, m, at);
    for (uint32_t i = 0; i < n && q + i < a.item_cap; i++)
        a.items[q + i] = make_uint4(l + i * ROW_ITEM, task, fits ? min(sz - i * ROW_ITEM, ROW_ITEM) | meta : 0u, ctx);
    return fits;
}

__global__ void __launch_bounds__(SWEEP_WARPS * 32, SWEEP_CTAS) k_sweep(const SweepArgs a)
{
    __shared__ SweepQueue queues[SWEEP_WARPS];
    if (*(volatile unsigned *)&a.ctl->error) return;   // (the batch check failed)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    SweepQueue &Q = queues[warp];
    uint32_t top = 0, rows = 0, windows = 0;   // intervals queued, their rows, windows queued
    uint32_t c_seeds = 0, c_verify = 0, c_vbytes = 0, c_vsect = 0;
    const uint64_t ntasks = 2 * a.rd.n;
    for (uint64_t base = ((uint64_t)blockIdx.x * SWEEP_WARPS + warp) * 32; base < ntasks;
         base += (uint64_t)gridDim.x * SWEEP_WARPS * 32) {
        const uint64_t t = base + (uint64_t)lane;
        const bool live = t < ntasks;
        const uint32_t rid = (uint32_t)(t >> 1), minus = (uint32_t)(t & 1);
        uint32_t m = 0, k = 0;
        const uint32_t *w = nullptr;
        if (live) {
            m = a.rd.len[rid];
            k = a.rd.k[rid];
            w = a.rd.words + a.rd.word_off[rid];
        }
        const uint32_t p = k + 1;
        const bool pieces = live && m >= p;
        // every scheme's table entries, all in flight together
        uint32_t code[4], l[4], r[4], qe[4];
#pragma unroll
        for (uint32_t j = 0; j < 4; j++) {
            l[j] = r[j] = code[j] = qe[j] = 0;
            if (pieces && j < p) {
                const uint32_t aj = bnd(j, m, p), bj = bnd(j + 1, m, p);
                qe[j] = min(a.seed.q, bj - aj);
                // P[bj - qe, bj) forward; of the other strand, R[m - bj, m - bj + qe) complemented
                const uint32_t s0 = minus ? m - bj : bj - qe[j], wi = s0 >> 4, o = s0 & 15u;
                const uint32_t lo = __ldg(w + wi), hi = o + qe[j] > 16u ? __ldg(w + wi + 1) : 0u;
                const uint32_t raw = __funnelshift_r(lo, hi, 2u * o) & ((1u << (2u * qe[j])) - 1u);
                code[j] = minus ? raw ^ ((1u << (2u * qe[j])) - 1u) : rev_groups(raw) >> (2u * (16u - qe[j]));
            }
        }
#pragma unroll
        for (uint32_t j = 0; j < 4; j++)
            if (qe[j]) {
                seed_interval_in(a.seed.table, a.seed.q, a.seed.nshort, a.seed.short_pad, a.seed.short_len,
                                 a.seed.short_bloom, code[j], qe[j], l[j], r[j]);
                c_seeds++;
            }
        uint32_t left = live && !pieces ? 1u : 0u;   // schemes for the bidirectional kernel
        const uint32_t jmax = __reduce_max_sync(SFULL, pieces ? p : 0u);
        // (not unrolled: four copies of what follows did not stay in the instruction cache)
#pragma unroll 1
        for (uint32_t j = 0; j < jmax; j++) {
            const uint32_t lj = j == 0 ? l[0] : j == 1 ? l[1] : j == 2 ? l[2] : l[3];
            const uint32_t rj = j == 0 ? r[0] : j == 1 ? r[1] : j == 2 ? r[2] : r[3];
            const uint32_t qj = j == 0 ? qe[0] : j == 1 ? qe[1] : j == 2 ? qe[2] : qe[3];
            const bool some = qj && lj < rj;
            const uint32_t sz = rj - lj;
            const bool rowwise = some && sz <= a.split_max && qj >= a.verify_min && m - qj >= BD_VERIFY_LEFT;
            const bool check = rowwise && sz <= a.split;
            const bool whole = some && qj == m;            // the seed is the whole read
            const bool larger = sweep_items(a, rowwise && !check, lj, sz, (uint32_t)t, w, m, k, j, qj, lane);
            if (some && !check && !whole && !larger) left |= 1u << j;
            sweep_emit(a, whole, rid, minus << 2, lj, rj, lane);
            const unsigned bal = __ballot_sync(SFULL, check);
            if (check) {
                const uint32_t q = top + __popc(bal & lt);
                const uint32_t at = bnd(j + 1, m, p) - qj;
                Q.iv[q] = make_uint4(lj, (uint32_t)t, sz | (j << 16) | (min(16u, at - bnd(j, m, p)) << 18) | (k << 23),
                                     read_context(w, minus, m, at));
                Q.at[q] = (uint16_t)at;
            }
            top += __popc(bal);
            rows += __reduce_add_sync(SFULL, check ? sz : 0u);
            __syncwarp();
            while (rows >= 32) {
                sweep_rows(a, Q, top, rows, windows, lane, c_vbytes, c_vsect);
                if (windows >= 32) sweep_windows(a, Q, windows, lane, c_verify, c_vbytes, c_vsect);
            }
        }
        const unsigned bal = __ballot_sync(SFULL, left != 0);
        if (bal) {
            unsigned long long at = 0;
            if (lane == 0) at = atomicAdd(&a.ctl->ntasks, (unsigned long long)__popc(bal));
            at = __shfl_sync(SFULL, at, 0) + __popc(bal & lt);
            if (left) a.list[at] = make_uint2((uint32_t)t, left);
        }
    }
    while (rows | windows) {
        if (rows) sweep_rows(a, Q, top, rows, windows, lane, c_vbytes, c_vsect);
        if (windows >= 32 || !rows) sweep_windows(a, Q, windows, lane, c_verify, c_vbytes, c_vsect);
    }
    c_seeds = __reduce_add_sync(SFULL, c_seeds);
    c_verify = __reduce_add_sync(SFULL, c_verify);
    c_vbytes = __reduce_add_sync(SFULL, c_vbytes);
    c_vsect = __reduce_add_sync(SFULL, c_vsect);
    if (lane == 0 && c_seeds) {
        atomicAdd(&a.ctl->seeds, (unsigned long long)c_seeds);
        atomicAdd(&a.ctl->verified, (unsigned long long)c_verify);
        atomicAdd(&a.ctl->verify_bytes, (unsigned long long)c_vbytes);
        atomicAdd(&a.ctl->verify_sectors, (unsigned long long)c_vsect);
    }
}

// One warp's windows of one read (starts st[0, n), n <= 32) against the text:
// four pattern words at a time, those of the exact piece first (most windows of
// a repeat family fail there).
__device__ __forceinline__ void item_windows(const SweepArgs &a, const uint32_t *pat, const uint32_t *st, uint32_t n,
                                             uint32_t rid, uint32_t minus, uint32_t m, uint32_t k, uint32_t j, int lane,
                                             uint32_t &c_verify, uint32_t &c_vbytes, uint32_t &c_vsect)
{
    const uint32_t p = k + 1;
    const uint32_t b1 = bnd(1, m, p), b2 = p >= 2 ? bnd(2, m, p) : 511u, b3 = p >= 3 ? bnd(3, m, p) : 511u;
    const uint32_t wn = (m + 15) >> 4, chunks = (wn + 3) >> 2, first = bnd(j, m, p) >> 6;
    bool live = (uint32_t)lane < n;
    const uint32_t s = live ? st[lane] : 0u;
    const uint32_t *tp = a.text + (s >> 4);
    const uint32_t sh = 2u * (s & 15u);
    uint32_t tot = 0, hit = 0;
    if (live) c_verify++;
    for (uint32_t i = 0; i < chunks; i++) {
        const uint32_t q0 = 4u * (first + i < chunks ? first + i : first + i - chunks);
        if (live) {
            uint32_t tw[5];
#pragma unroll
            for (uint32_t u = 0; u < 5; u++) tw[u] = q0 + u <= wn ? __ldg(tp + q0 + u) : 0u;
            c_vbytes += 4u * (min(4u, wn - q0) + 1u);
            c_vsect += ((((s >> 4) + q0) & 7u) * 4u + 4u * min(4u, wn - q0) + 35u) / 32u;
#pragma unroll
            for (uint32_t u = 0; u < 4; u++) {
                const uint32_t q = q0 + u;
                uint32_t x = pat[min(q, MAX_WORDS - 1)] ^ __funnelshift_r(tw[u], tw[u + 1], sh);
                x = (x | (x >> 1)) & 0x55555555u & low_mask(2u * (uint32_t)min(max((int)m - 16 * (int)q, 0), 16));
                while (x && tot <= k) {
                    const uint32_t pos = 16u * q + (uint32_t)(__ffs(x) - 1) / 2u;
                    x &= x - 1;
                    tot++;
                    hit |= 1u << ((pos >= b1) + (pos >= b2) + (pos >= b3));
                }
            }
            live = tot <= k && !((hit >> j) & 1u);
        }
        if (!__any_sync(SFULL, live)) return;
    }
    const bool leaf = live && (hit & ((1u << j) - 1u)) == (1u << j) - 1u;
    const unsigned bal = __ballot_sync(SFULL, leaf);
    if (!bal) return;
    uint32_t at = 0;
    if (lane == 0) {
        at = atomicAdd(&a.ctl->iv_count, (unsigned)__popc(bal));
        atomicAdd(&a.iv_cnt[rid], (unsigned)__popc(bal));
    }
    at = __shfl_sync(SFULL, at, 0) + __popc(bal & ((1u << lane) - 1u));
    if (leaf) {
        if (at < a.ctl->iv_cap) {
            Interval x;
            x.read = rid; x.meta = tot | (minus << 2) | IV_POS; x.l = s; x.r = s + 1u;
            a.iv[at] = x;
        } else {
            atomicOr(&a.ctl->error, ERR_IV_OVERFLOW);
        }
    }
}

// The item list, one item of one read per warp at a time: its rows stream by
// 32 at a time, those whose left context passes are collected and checked
// against the text 32 at a time, with the pattern in shared memory.  Intervals
// of this size come from repeats, a few thousand reads of a batch: here they
// spread over every warp of the GPU, where the sweep's own warps would each
// be held by the few they drew.
__global__ void __launch_bounds__(SWEEP_WARPS * 32, SWEEP_CTAS) k_rows(const SweepArgs a)
{
    __shared__ uint32_t pat_s[SWEEP_WARPS][MAX_WORDS], start_s[SWEEP_WARPS][64];
    const uint32_t n_items = min(*(volatile unsigned *)&a.ctl->row_items, a.item_cap);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t *pat = pat_s[warp], *st = start_s[warp];
    uint32_t c_verify = 0, c_vbytes = 0, c_vsect = 0;
    for (uint32_t it = blockIdx.x * SWEEP_WARPS + warp; it < n_items; it += gridDim.x * SWEEP_WARPS) {
        const uint4 item = __ldg(a.items + it);
        const uint32_t cnt = item.z & 511u, j = (item.z >> 9) & 3u, ex = (item.z >> 11) & 31u, k = (item.z >> 16) & 3u;
        const uint32_t at = item.z >> 18, rid = item.y >> 1, minus = item.y & 1u;
        if (cnt == 0) continue;
        const uint32_t m = a.rd.len[rid];
        const int wn = (int)((m + 15) >> 4);
        const uint32_t *w = a.rd.words + a.rd.word_off[rid];
        if (lane < (int)MAX_WORDS)
            pat[lane] = minus ? rc_word(raw_word(w, wn - 1 - lane, wn), raw_word(w, wn - 2 - lane, wn), m)
                              : raw_word(w, lane, wn);
        __syncwarp();
        uint32_t have = 0;
        for (uint32_t r0 = 0; r0 < cnt; r0 += 32) {
            bool stay = false;
            uint32_t s = 0;
            if (r0 + (uint32_t)lane < cnt) {
                const uint2 x = __ldg(a.sa_ctx + item.x + r0 + (uint32_t)lane);
                s = x.x - at;
                uint32_t df = x.y ^ item.w;
                df = (df | (df >> 1)) & 0x55555555u;
                if (at < 16u) df &= at ? ~0u << (2u * (16u - at)) : 0u;
                const bool exact = ex == 0 || (df >> (2u * (16u - ex))) == 0;
                stay = x.x >= at && (uint64_t)s + m <= a.n && exact && __popc(df) <= k;
                c_vbytes += 8u;
                c_vsect += (lane & 3) == 0;
            }
            const unsigned bal = __ballot_sync(SFULL, stay);
            if (stay) st[have + __popc(bal & ((1u << lane) - 1u))] = s;
            have += __popc(bal);
            __syncwarp();
            if (have >= 32u) {
                item_windows(a, pat, st, 32u, rid, minus, m, k, j, lane, c_verify, c_vbytes, c_vsect);
                have -= 32u;
                const uint32_t rest = (uint32_t)lane < have ? st[32 + lane] : 0u;
                __syncwarp();
                if ((uint32_t)lane < have) st[lane] = rest;
                __syncwarp();
            }
        }
        if (have) item_windows(a, pat, st, have, rid, minus, m, k, j, lane, c_verify, c_vbytes, c_vsect);
        __syncwarp();
    }
    c_verify = __reduce_add_sync(SFULL, c_verify);
    c_vbytes = __reduce_add_sync(SFULL, c_vbytes);
    c_vsect = __reduce_add_sync(SFULL, c_vsect);
    if (lane == 0 && c_vbytes) {
        atomicAdd(&a.ctl->verified, (unsigned long long)c_verify);
        atomicAdd(&a.ctl->verify_bytes, (unsigned long long)c_vbytes);
        atomicAdd(&a.ctl->verify_sectors, (unsigned long long)c_vsect);
    }
}

}  // namespace

// Rows of an interval the sweep checks itself, and those it puts on the item
// list.  Up to 32 are a warp's one look.  Past 256 a read's hits outgrow the
// warp that finishes it: us per pass with 32 (no list) / 128 / 256 / 512 / 1024
// / 2048, 64 Mbp 1M reads 1378 / 1308 / 1233 / 1225 / 1299 / 1520, uneven 1M 2506
// / 2428 / 2290 / 2272 / 2404 / 3416, 33k short reads with a cap of 10 313 / 309
// / 296 / 349 / 334 / 335, a human-like genome within 2%.
constexpr uint32_t SWEEP_SPLIT = 32;
constexpr uint32_t SWEEP_SPLIT_MAX = 256;

// May the sweep run for an index and its verify threshold (matched bases)?
// It needs the suffix array and the text, and seeds long enough to be checked.
bool sweep_available(const mica_index *idx, uint32_t verify_min)
{
    const uint32_t q = idx->view.lfwd.table ? idx->view.lfwd.q : idx->view.q;
    return idx->view.sa_ctx && verify_min && verify_min <= q;
}

// Enqueue the sweep of n reads: leaves into iv, the tasks left into list (2 n
// entries), their number in ctl->ntasks (0 before).
int enqueue_sweep(const mica_index *idx, Workspace &w, const ReadsView &rd, uint32_t verify_min, uint32_t budget, uint2 *list,
                  uint4 *items, uint32_t item_cap, cudaStream_t s, uint64_t &launches)
{
    SweepArgs a{};
    const IndexView &v = idx->view;
    if (v.lfwd.table) {
        a.seed = v.lfwd;
    } else {
        a.seed.table = v.table;
        a.seed.q = v.q;
        a.seed.nshort = v.nshort;
        a.seed.short_bloom = v.short_bloom;
        for (uint32_t i = 0; i < MAX_Q; i++) {
            a.seed.short_pad[i] = v.short_pad[i];
            a.seed.short_len[i] = v.short_len[i];
        }
    }
    a.sa_ctx = v.sa_ctx;
    a.text = v.text;
    a.n = v.n;
    a.rd = rd;
    a.ctl = (SearchCtl *)w.ctl.p;
    a.iv = (Interval *)w.iv.p;
    a.iv_cnt = (uint32_t *)w.iv_cnt.p;
    a.list = list;
    a.verify_min = verify_min;
    a.split = SWEEP_SPLIT;
    // (a node budget below 64 asks for short turns: then larger intervals stay with the tree, which it governs)
    a.split_max = budget < 64 ? SWEEP_SPLIT : SWEEP_SPLIT_MAX;
    a.items = items;
    a.item_cap = item_cap;
    const uint64_t blocks = (2 * rd.n + SWEEP_WARPS * 32 - 1) / (SWEEP_WARPS * 32);
    k_sweep<<<(unsigned)std::min<uint64_t>(blocks, 152ull * SWEEP_CTAS), SWEEP_WARPS * 32, 0, s>>>(a);
    k_rows<<<152 * SWEEP_CTAS, SWEEP_WARPS * 32, 0, s>>>(a);
    launches += 2;
    MICA_CUDA_TRY(cudaGetLastError());
    return 0;
}

}  // namespace mica

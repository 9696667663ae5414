// The seed sweep: the first pass of the bidirectional search (bidir.cu).  With
// the whole suffix array and the text resident it also checks rows; without them
// it only makes every seed the first node of a tree.
//
// Most schemes of most reads need no search tree: the exact piece's last q
// bases come up empty in the seed table (a read's other strand, mostly) or
// name a few rows, each of which one look at the text decides.  The sweep does
// exactly those: one thread per (read, strand) looks its k + 1 seeds up, the
// rows of the small intervals are checked against the text 32 at a time, those
// of somewhat larger ones go on a list (k_rows), and only the schemes it cannot
// finish (an interval of many rows, a piece too short to be told apart, a read
// shorter than k + 1 bases) become trees (tree.cu), or, when a small node budget
// is set or the frontier is full, tasks with a bit per scheme for bidir.cu's
// kernel.
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
// Mbp genome with repeats: 1.57 ms before, 0.93 ms now, 0.49 ms of it the sweep
// (6M seeds and 3M rows at 30 G random reads/s would take 0.3 ms).
#include <algorithm>

#include "sweep_common.cuh"

namespace mica {
namespace {

constexpr unsigned SFULL = 0xffffffffu;
constexpr int SWEEP_WARPS = 8;
constexpr int SWEEP_CTAS = 4;     // per SM
constexpr uint32_t ROWS_SMALL = 16;   // rows of an item that shares a warp's look with others
constexpr int SWEEP_QUEUE = 64;   // intervals waiting: fewer than 32 left over (each has a row) plus 32 new ones

struct SweepArgs {
    QmerView seed, rseed;        // the longer tables of G$ and G~$ when there are such
    uint4 *nodes;                // the trees' first frontier (null: everything left goes on the list)
    uint32_t *node_meta;
    uint32_t node_cap;
    uint32_t rows_all;           // N + 1
    const uint2 *sa_ctx;
    const uint32_t *text;
    uint64_t n;
    ReadsView rd;
    SearchCtl *ctl;
    Interval *iv;
    uint32_t *iv_cnt;
    uint2 *list;                 // (task, schemes left as bits)
    // larger intervals (sweep_common.cuh)
    uint4 *items;
    uint32_t item_cap;
    uint32_t verify_min, split, split_max;
};

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

// Put the warp's larger intervals (lanes with `want`) on the item list, with
// one counter update; false for a lane past the list's end (the counter then
// stays above it, and item_cap is what k_rows and the trees go by too, so that
// no entry that nobody wrote is read).
__device__ __forceinline__ bool sweep_items(const SweepArgs &a, bool want, uint32_t l, uint32_t sz, uint32_t task,
                                            const uint32_t *w, uint32_t m, uint32_t k, uint32_t j, uint32_t qe,
                                            int lane)
{
    const unsigned bal = __ballot_sync(SFULL, want);
    if (!bal) return false;
    uint32_t q = 0;
    if (lane == 0) q = atomicAdd(&a.ctl->row_items, (unsigned)__popc(bal));
    q = __shfl_sync(SFULL, q, 0) + __popc(bal & ((1u << lane) - 1u));
    if (!want || q >= a.item_cap) return false;
    const uint32_t at = bnd(j + 1, m, k + 1) - qe;
    a.items[q] = make_uint4(l, task, item_meta(sz, j, min(16u, at - bnd(j, m, k + 1)), k, at, k),
                            read_context(w, task & 1u, m, at));
    return true;
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
            const bool rowwise = some && a.verify_min && sz <= a.split_max && qj >= a.verify_min && m - qj >= BD_VERIFY_LEFT;
            const bool check = rowwise && sz <= a.split;
            const bool whole = some && qj == m;            // the seed is the whole read
            const bool larger = sweep_items(a, rowwise && !check, lj, sz, (uint32_t)t, w, m, k, j, qj, lane);
            const bool grow = some && !check && !whole && !larger;
            if (a.nodes) {
                // the tree's first node: the reversed seed's interval in the reversed genome's index too
                const unsigned bal = __ballot_sync(SFULL, grow);
                if (bal) {
                    unsigned long long at = 0;
                    if (lane == 0) at = atomicAdd(&a.ctl->ntasks, (unsigned long long)__popc(bal));
                    at = __shfl_sync(SFULL, at, 0) + __popc(bal & lt);
                    if (grow && at < a.node_cap) {
                        const uint32_t cj = j == 0 ? code[0] : j == 1 ? code[1] : j == 2 ? code[2] : code[3];
                        uint32_t lr, rr;
                        seed_interval_in(a.rseed.table, a.rseed.q, a.rseed.nshort, a.rseed.short_pad, a.rseed.short_len,
                                         a.rseed.short_bloom, rev_groups(cj) >> (2u * (16u - qj)), qj, lr, rr);
                        c_seeds++;
                        const uint32_t bj = bnd(j + 1, m, p);
                        a.nodes[at] = make_uint4((uint32_t)t, lj, lr, sz);
                        a.node_meta[at] = bd_meta(0, bj - qj, bj, 0, 0, j);
                    } else if (grow) {
                        left |= 1u << j;
                    }
                }
            } else if (grow) {
                left |= 1u << j;
            }
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
        if (a.nodes) {
            // a read shorter than k + 1 bases: the whole tree from the full interval
            const bool full = left && !pieces;
            const unsigned bal = __ballot_sync(SFULL, full);
            if (bal) {
                unsigned long long at = 0;
                if (lane == 0) at = atomicAdd(&a.ctl->ntasks, (unsigned long long)__popc(bal));
                at = __shfl_sync(SFULL, at, 0) + __popc(bal & lt);
                if (full && at < a.node_cap) {
                    a.nodes[at] = make_uint4((uint32_t)t, 0u, 0u, a.rows_all);
                    a.node_meta[at] = bd_meta(0, m, m, 0, 0, SCHEME_FREE);
                    left = 0;
                }
            }
        }
        const unsigned bal = __ballot_sync(SFULL, left != 0);
        if (bal) {
            unsigned long long at = 0;
            if (lane == 0)
                at = atomicAdd(a.nodes ? &a.ctl->pool_tasks : &a.ctl->ntasks, (unsigned long long)__popc(bal));
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

// One item of many rows: they stream by 32 at a time, those whose left context
// passes are collected in st and checked against the text 32 at a time, with
// the pattern in shared memory (pat).
__device__ __forceinline__ void rows_of_item(const SweepArgs &a, const uint4 item, uint32_t *pat, uint32_t *st, int lane,
                                             uint32_t &c_verify, uint32_t &c_vbytes, uint32_t &c_vsect)
{
    const uint32_t cnt = item.z & 511u, j = (item.z >> 9) & 3u, ex = (item.z >> 11) & 31u, k = (item.z >> 16) & 3u;
    const uint32_t at = (item.z >> 18) & 511u, rem = (item.z >> 27) & 3u, rid = item.y >> 1, minus = item.y & 1u;
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
            stay = x.x >= at && (uint64_t)s + m <= a.n && exact && __popc(df) <= rem;
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

// The item list.  Items of many rows come from repeats, a few thousand reads of
// a batch: they spread over every warp of the GPU, one at a time, where the
// sweep's own warps would each be held by the few they drew.  A tree's items
// are mostly of a row or a few, and millions when its seeds are short: a warp
// takes up to 32 of them and looks at the rows of several together, as the
// sweep does.  (A warp for each of those too took 2.4 ms for 100k reads of 30
// bp, k = 2, on a 16 Mbp genome, this way 0.65.)
__global__ void __launch_bounds__(SWEEP_WARPS * 32, SWEEP_CTAS) k_rows(const SweepArgs a)
{
    __shared__ uint32_t pat_s[SWEEP_WARPS][MAX_WORDS], start_s[SWEEP_WARPS][64];
    __shared__ SweepQueue queues[SWEEP_WARPS];
    const uint32_t n_items = min(*(volatile unsigned *)&a.ctl->row_items, a.item_cap);
    if (n_items == 0 || *(volatile unsigned *)&a.ctl->error) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    SweepQueue &Q = queues[warp];
    uint32_t c_verify = 0, c_vbytes = 0, c_vsect = 0;
    uint32_t top = 0, rows = 0, windows = 0;   // small items queued, their rows, windows queued
    // (few items: one at a time, so that neighbours on the list, one repeat's, spread over the warps;
    // with at least 1 / 8 / 32 turns a warp repeats_1m 1.26 / 1.19 / 1.18 ms, uneven_1m 2.11 / 2.07 / 1.99)
    const uint32_t warps = gridDim.x * SWEEP_WARPS, per = max(1u, min(32u, n_items / (warps * 32u)));
    for (uint64_t i0 = (uint64_t)(blockIdx.x * SWEEP_WARPS + warp) * per; i0 < n_items; i0 += (uint64_t)warps * per) {
        uint4 item = make_uint4(0, 0, 0, 0);
        const bool has = (uint32_t)lane < per && i0 + (uint32_t)lane < n_items;
        if (has) item = __ldg(a.items + i0 + (uint32_t)lane);
        const uint32_t cnt = item.z & 511u;
        const bool small = has && cnt <= ROWS_SMALL;
        for (unsigned big = __ballot_sync(SFULL, has && !small); big; big &= big - 1) {
            const int src = __ffs(big) - 1;
            rows_of_item(a, make_uint4(__shfl_sync(SFULL, item.x, src), __shfl_sync(SFULL, item.y, src),
                                       __shfl_sync(SFULL, item.z, src), __shfl_sync(SFULL, item.w, src)),
                         pat_s[warp], start_s[warp], lane, c_verify, c_vbytes, c_vsect);
        }
        const unsigned bal = __ballot_sync(SFULL, small);
        if (small) {
            const uint32_t q = top + __popc(bal & lt);
            Q.iv[q] = make_uint4(item.x, item.y, cnt | (((item.z >> 9) & 3u) << 16) | (((item.z >> 11) & 31u) << 18) |
                                 (((item.z >> 27) & 3u) << 23), item.w);
            Q.at[q] = (uint16_t)((item.z >> 18) & 511u);
        }
        top += __popc(bal);
        rows += __reduce_add_sync(SFULL, small ? cnt : 0u);
        __syncwarp();
        while (rows >= 32) {
            sweep_rows(a, Q, top, rows, windows, lane, c_vbytes, c_vsect);
            if (windows >= 32) sweep_windows(a, Q, windows, lane, c_verify, c_vbytes, c_vsect);
        }
    }
    while (rows | windows) {
        if (rows) sweep_rows(a, Q, top, rows, windows, lane, c_vbytes, c_vsect);
        if (windows >= 32 || !rows) sweep_windows(a, Q, windows, lane, c_verify, c_vbytes, c_vsect);
    }
    c_verify = __reduce_add_sync(SFULL, c_verify);
    c_vbytes = __reduce_add_sync(SFULL, c_vbytes);
    c_vsect = __reduce_add_sync(SFULL, c_vsect);
    if (lane == 0 && c_vbytes) {
        atomicAdd(&a.ctl->verified, (unsigned long long)c_verify);
        atomicAdd(&a.ctl->verify_bytes, (unsigned long long)c_vbytes);
        atomicAdd(&a.ctl->verify_sectors, (unsigned long long)c_vsect);
    }
    // the last CTA: the list is empty again (a search may go on and add to it)
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&a.ctl->done_rows, 1u) == gridDim.x - 1) {
        a.ctl->row_items = 0;
        a.ctl->done_rows = 0;
    }
}

}  // namespace

// Rows of an interval the sweep checks itself, and those it puts on the item
// list.  Up to 32 are a warp's one look; past 64 a first extension in the trees
// drops most rows of a repeat family for less than their checks cost (32 / 64 /
// 128 / 256, when k_rows gave each item a warp: 512 Mbp human-like 1M mates 3.57 /
// 3.57 / 3.58 / 4.00 ms of search kernels, uneven 1M reads 1.38 / 1.39 / 1.50 / 1.55).
constexpr uint32_t SWEEP_SPLIT = 32;
constexpr uint32_t SWEEP_SPLIT_MAX = 64;

static void base_view(QmerView &q, const uint32_t *table, uint32_t len, uint32_t nshort, const uint32_t *pad,
                      const uint32_t *slen, unsigned long long bloom)
{
    q.table = table;
    q.q = len;
    q.nshort = nshort;
    q.short_bloom = bloom;
    for (uint32_t i = 0; i < MAX_Q; i++) {
        q.short_pad[i] = pad[i];
        q.short_len[i] = slen[i];
    }
}

static SweepArgs sweep_args(const mica_index *idx, Workspace &w, const ReadsView &rd)
{
    SweepArgs a{};
    const IndexView &v = idx->view;
    if (v.lfwd.table) {
        a.seed = v.lfwd;
        a.rseed = v.lrev;
    } else {
        base_view(a.seed, v.table, v.q, v.nshort, v.short_pad, v.short_len, v.short_bloom);
        base_view(a.rseed, v.rev.table, v.q, v.rev.nshort, v.rev.short_pad, v.rev.short_len, v.rev.short_bloom);
    }
    a.sa_ctx = v.sa_ctx;
    a.text = v.text;
    a.n = v.n;
    a.rows_all = v.rows;
    a.rd = rd;
    a.ctl = (SearchCtl *)w.ctl.p;
    a.iv = (Interval *)w.iv.p;
    a.iv_cnt = (uint32_t *)w.iv_cnt.p;
    return a;
}

// Enqueue the sweep of n reads: leaves into iv, larger intervals' rows into
// items, and what is left as nodes (up to `cap`, their number in ctl->ntasks,
// 0 before), or, with none given or past their end, as tasks with a bit per
// scheme in list (2 n entries; ctl->pool_tasks, or ctl->ntasks without nodes).
int enqueue_sweep(const mica_index *idx, Workspace &w, const ReadsView &rd, uint32_t verify_min, uint32_t budget,
                  uint2 *list, uint4 *nodes, uint32_t *node_meta, uint32_t cap, uint4 *items, uint32_t item_cap,
                  cudaStream_t s, uint64_t &launches)
{
    SweepArgs a = sweep_args(idx, w, rd);
    a.list = list;
    a.nodes = nodes;
    a.node_meta = node_meta;
    a.node_cap = cap;
    a.items = items;
    a.item_cap = item_cap;
    a.verify_min = verify_min;
    a.split = SWEEP_SPLIT;
    // (a node budget below 64 asks for short turns: then larger intervals stay with the tree, which it governs)
    a.split_max = budget && budget < 64 ? SWEEP_SPLIT : SWEEP_SPLIT_MAX;
    const uint64_t blocks = (2 * rd.n + SWEEP_WARPS * 32 - 1) / (SWEEP_WARPS * 32);
    k_sweep<<<(unsigned)std::min<uint64_t>(blocks, 152ull * SWEEP_CTAS), SWEEP_WARPS * 32, 0, s>>>(a);
    launches++;
    MICA_CUDA_TRY(cudaGetLastError());
    return 0;
}

// Enqueue the check of the items not yet done.
int enqueue_rows(const mica_index *idx, Workspace &w, const ReadsView &rd, uint4 *items, uint32_t item_cap,
                 cudaStream_t s, uint64_t &launches)
{
    SweepArgs a = sweep_args(idx, w, rd);
    a.items = items;
    a.item_cap = item_cap;
    k_rows<<<152 * SWEEP_CTAS, SWEEP_WARPS * 32, 0, s>>>(a);
    launches++;
    MICA_CUDA_TRY(cudaGetLastError());
    return 0;
}

}  // namespace mica

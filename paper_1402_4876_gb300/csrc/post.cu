// From leaf SA intervals to per-read hit lists, in five kernels (seven for more
// than 512 reads):
//   1. k_tile_counts, k_offsets: prefix sum of the per-read interval counts;
//   2. k_iv_scatter: the intervals grouped by read, and total = the sum of a
//      read's interval sizes (exact), of which min(total, cap) rows are listed;
//   3. k_listed: the rows listed per tile of reads;
//   4. k_finish_small: prefix sum of the listed counts -> CSR offsets, and the
//      hits of reads with a few; larger reads and reads over their cap go on
//      lists;
//   5. k_finish_block (blocks of two sizes): those reads, a warp or a block each: over
//      the cap the first cap rows in the order (d, strand, row) are kept, then
//      rows become text positions, and the hits go out sorted by (position,
//      strand).
// A row's position is one read of the suffix array when the index keeps it,
// else LF walks to the nearest marked row (SA[j] % s == 0), whose SA value is
// stored: SA[j] = SA[LF^t(j)] + t, LF(j) = C[BWT[j]] + Occ(BWT[j], j).
//
// The first form of this had a kernel per step over all hits (fourteen
// launches, each hit written, located and sorted in global memory); with the
// hits of a read made, ordered and written in one place each is written once.
#include <stddef.h>

#include <algorithm>
#include <vector>

#include "search_common.cuh"

namespace mica {

namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;
constexpr unsigned FULL = 0xffffffffu;
constexpr uint32_t TILE = 512;                // reads per block of the per-read passes
constexpr uint32_t TILE_THREADS = 256;
constexpr uint64_t SCAN_TILES = 16384;        // more tiles than this: their sums are scanned by a kernel
constexpr uint32_t SMALL_HITS = 8;             // reads up to this many hits: one thread each
constexpr uint32_t WARP_HITS = 256;            // up to this many hits and intervals: a warp each
constexpr uint32_t WARP_CAP = 65535;           // (and a cap its 32-bit sums hold)
constexpr uint32_t BLOCK_HITS = 4096;          // up to this many hits: a block each; above: the host's loop
constexpr uint32_t BLOCK_READ_THREADS = 128;
constexpr uint32_t LONG_LIST = 1024;           // a read of more intervals than this has a block ...
constexpr uint32_t LONG_THREADS = 1024;        // ... of this many threads
constexpr uint32_t WARP_SPAN = 4096;           // hits within this many positions of each other are ordered by counting:
constexpr uint32_t BLOCK_SPAN = 20480;         // a bit per (position, strand) in shared memory

// ---- exclusive scan (n values -> n + 1 offsets) ----

template <typename T>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_tiles(const T *__restrict__ in, uint64_t n,
                                                             uint64_t *__restrict__ out,
                                                             uint64_t *__restrict__ tile_sums)
{
    __shared__ uint64_t warp_sums[SCAN_THREADS / 32];
    uint64_t base = (uint64_t)blockIdx.x * SCAN_TILE + threadIdx.x * SCAN_ITEMS;
    uint64_t v[SCAN_ITEMS];
    uint64_t sum = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        v[j] = (base + j < n) ? (uint64_t)in[base + j] : 0ull;
        sum += v[j];
    }
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint64_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    uint64_t woff = 0, total = 0;
    for (int w = 0; w < SCAN_THREADS / 32; w++) {
        if (w < warp) woff += warp_sums[w];
        total += warp_sums[w];
    }
    uint64_t run = woff + incl - sum;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        if (base + j < n) out[base + j] = run;
        run += v[j];
    }
    if (threadIdx.x == 0) tile_sums[blockIdx.x] = total;
}

// one block: exclusive scan of the tile sums, grand total at [ntiles]
__global__ void __launch_bounds__(1024) k_scan_sums(uint64_t *__restrict__ s, uint64_t ntiles)
{
    __shared__ uint64_t warp_sums[32];
    __shared__ uint64_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (uint64_t b0 = 0; b0 < ntiles; b0 += 1024) {
        uint64_t i = b0 + threadIdx.x;
        uint64_t x = i < ntiles ? s[i] : 0;
        uint64_t incl = x;
        for (int o = 1; o < 32; o <<= 1) {
            uint64_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) warp_sums[warp] = incl;
        __syncthreads();
        uint64_t woff = 0, tot = 0;
        for (int w = 0; w < 32; w++) {
            if (w < warp) woff += warp_sums[w];
            tot += warp_sums[w];
        }
        uint64_t c = carry;
        if (i < ntiles) s[i] = c + woff + incl - x;
        __syncthreads();
        if (threadIdx.x == 0) carry = c + tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) s[ntiles] = carry;
}

__global__ void k_scan_add(uint64_t *__restrict__ out, uint64_t n, const uint64_t *__restrict__ tile_sums)
{
    uint64_t ntiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x)
        out[i] += tile_sums[i / SCAN_TILE];
    if (blockIdx.x == 0 && threadIdx.x == 0) out[n] = tile_sums[ntiles];
}

// ---- per-read prefix sums: a block per tile of reads, which adds up the tiles before its own ----

__device__ __forceinline__ uint64_t block_exclusive(uint64_t v, uint64_t *warp_sums, uint64_t &all)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
    }
    __syncthreads();
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    uint64_t before = 0;
    all = 0;
    for (uint32_t w = 0; w < TILE_THREADS / 32; w++) {
        if ((int)w < warp) before += warp_sums[w];
        all += warp_sums[w];
    }
    return before + incl - v;
}

// Sum of the first `tiles` tile sums, which every block reads: few loads for a
// million reads, but they grow with the square.  Above SCAN_TILES a kernel of
// one block scans the sums first: the kernels after the search without / with it
// 120 / 127 us for 2M reads, 406 / 409 for 8M, 898 / 811 for 16M.
__device__ __forceinline__ uint64_t tiles_before(const uint64_t *__restrict__ sums, uint32_t tiles, uint64_t *warp_sums)
{
    uint64_t v = 0, all;
    for (uint32_t i = threadIdx.x; i < tiles; i += TILE_THREADS) v += sums[i];
    block_exclusive(v, warp_sums, all);
    return all;
}

__global__ void __launch_bounds__(TILE_THREADS) k_tile_counts(const uint32_t *__restrict__ cnt, uint64_t n,
                                                              uint64_t *__restrict__ sums)
{
    __shared__ uint64_t ws[TILE_THREADS / 32];
    uint64_t v = 0, all;
    for (uint32_t i = threadIdx.x; i < TILE; i += TILE_THREADS) {
        const uint64_t r = blockIdx.x * (uint64_t)TILE + i;
        if (r < n) v += cnt[r];
    }
    block_exclusive(v, ws, all);
    if (threadIdx.x == 0) sums[blockIdx.x] = all;
}

// off[r] = sum of cnt[0, r), r = 0 .. n, and total[r] = 0.  sums: of the tiles
// before (not read by the first), each alone or (scanned) all before it.
__global__ void __launch_bounds__(TILE_THREADS) k_offsets(const uint32_t *__restrict__ cnt, uint64_t n,
                                                          const uint64_t *__restrict__ sums, bool scanned,
                                                          uint64_t *__restrict__ off, uint64_t *__restrict__ total)
{
    __shared__ uint64_t ws[TILE_THREADS / 32];
    uint64_t at = scanned ? sums[blockIdx.x] : tiles_before(sums, blockIdx.x, ws);
    constexpr uint32_t PER = TILE / TILE_THREADS;
    const uint64_t r0 = blockIdx.x * (uint64_t)TILE + threadIdx.x * PER;
    uint32_t c[PER];
    uint64_t v = 0, all;
#pragma unroll
    for (uint32_t i = 0; i < PER; i++) {
        c[i] = r0 + i < n ? cnt[r0 + i] : 0u;
        v += c[i];
    }
    at += block_exclusive(v, ws, all);
#pragma unroll
    for (uint32_t i = 0; i < PER; i++) {
        if (r0 + i <= n) off[r0 + i] = at;
        if (r0 + i < n) total[r0 + i] = 0;
        at += c[i];
    }
    // (the last read's thread writes off[n] above unless n ends a tile)
    if (r0 + PER == n) off[n] = at;
}

// ---- intervals grouped by read ----

// Every post kernel that indexes by the search's per-read counts first looks
// at how the search ended: after an overflow the counts exceed what was
// stored, and after rounds that left nodes or gave reads up they are not
// complete.  Then these kernels do nothing, and the caller finishes the
// search or runs it again before it calls them again.
__device__ __forceinline__ bool search_open(const SearchCtl *ctl)
{
    return (*(const volatile unsigned *)&ctl->error | *(const volatile unsigned *)&ctl->unfinished) != 0;
}

// The interval count is read on the device (capped at the buffer's capacity) so
// the launch needs no host round trip.
__global__ void k_iv_scatter(const Interval *__restrict__ iv, const SearchCtl *__restrict__ ctl, uint32_t cap, const uint64_t *__restrict__ iv_off, uint32_t *__restrict__ cursor,
                             Interval *__restrict__ out, unsigned long long *__restrict__ total)
{
    if (search_open(ctl)) return;
    const uint32_t count = min(ctl->iv_count, cap);
    for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < count; e += gridDim.x * blockDim.x) {
        Interval x = iv[e];
        if (x.read == IV_PURGED) continue;   // a leaf of a read that was searched again
        uint32_t at = atomicSub(&cursor[x.read], 1u) - 1u;
        out[iv_off[x.read] + at] = x;
        atomicAdd(&total[x.read], (unsigned long long)(x.r - x.l));
    }
}

// An interval in rows: a text position found by the text check becomes its
// row (only a capped read's order needs it).
__device__ __forceinline__ void to_rows(Interval &x, const uint32_t *__restrict__ isa)
{
    if (x.meta & IV_POS) {
        x.l = __ldg(isa + x.l);
        x.r = x.l + 1u;
        x.meta &= ~IV_POS;
    }
}

__device__ __forceinline__ uint64_t iv_key(const Interval &x)
{
    return ((uint64_t)(x.meta & 3u) << 33) | ((uint64_t)((x.meta >> 2) & 1u) << 32) | x.l;
}

// The tile's listed hits, min(total, cap) per read, to sums.
__global__ void __launch_bounds__(TILE_THREADS) k_listed(const uint64_t *__restrict__ total, uint64_t n, uint32_t cap,
                                                         uint64_t *__restrict__ sums)
{
    __shared__ uint64_t ws[TILE_THREADS / 32];
    uint64_t keep = 0, all;
    for (uint32_t i = threadIdx.x; i < TILE; i += TILE_THREADS) {
        const uint64_t r = blockIdx.x * (uint64_t)TILE + i;
        const uint64_t t = r < n ? total[r] : 0;
        keep += cap && t > cap ? cap : t;
    }
    block_exclusive(keep, ws, all);
    if (threadIdx.x == 0) sums[blockIdx.x] = all;
}

// Best-stratum reporting: a read keeps only its intervals with the smallest
// d; the others become empty (r = l) and so count and list nothing.  A read
// with many intervals is gone through by its warp.
__global__ void k_stratum(Interval *__restrict__ ivs, const uint64_t *__restrict__ iv_off, uint64_t n,
                          uint64_t *__restrict__ total, const SearchCtl *__restrict__ ctl)
{
    if (search_open(ctl)) return;
    const uint32_t lane = threadIdx.x & 31;
    for (uint64_t r0 = blockIdx.x * (uint64_t)blockDim.x + (threadIdx.x & ~31u); r0 < n;
         r0 += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t r = r0 + lane;
        uint64_t b = 0, e = 0;
        if (r < n) { b = iv_off[r]; e = iv_off[r + 1]; }
        const bool many = e - b > 32;
        if (!many && e - b > 1) {
            uint32_t dmin = 3;
            uint64_t gone = 0;
            for (uint64_t x = b; x < e; x++) dmin = min(dmin, ivs[x].meta & 3u);
            for (uint64_t x = b; x < e; x++) {
                const Interval v = ivs[x];
                if ((v.meta & 3u) > dmin) { ivs[x].r = v.l; gone += v.r - v.l; }
            }
            if (gone) total[r] -= gone;
        }
        for (unsigned todo = __ballot_sync(FULL, many); todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const uint64_t wb = __shfl_sync(FULL, b, src), we = __shfl_sync(FULL, e, src);
            uint32_t dmin = 3;
            for (uint64_t x = wb + lane; x < we; x += 32) dmin = min(dmin, ivs[x].meta & 3u);
            dmin = __reduce_min_sync(FULL, dmin);
            uint64_t gone = 0;
            for (uint64_t x = wb + lane; x < we; x += 32) {
                const Interval v = ivs[x];
                if ((v.meta & 3u) > dmin) { ivs[x].r = v.l; gone += v.r - v.l; }
            }
            for (int o = 16; o; o >>= 1) gone += __shfl_xor_sync(FULL, gone, o);
            if ((int)lane == src) total[r] -= gone;
        }
    }
}

// Sum of all tile sums (the hits to be listed), for the host.
__global__ void __launch_bounds__(TILE_THREADS) k_tiles_total(const uint64_t *__restrict__ sums, uint32_t tiles,
                                                              uint64_t *__restrict__ out)
{
    __shared__ uint64_t ws[TILE_THREADS / 32];
    const uint64_t all = tiles_before(sums, tiles, ws);
    if (threadIdx.x == 0) *out = all;
}

}  // namespace

// ---- locate: SA[j] by LF walks to a marked row ----

__device__ __forceinline__ uint32_t locate_row(const IndexView &ix, uint32_t j, uint32_t &steps)
{
    uint32_t t = 0;
    for (;;) {
        uint32_t mb = j / MARK_ROWS, mo = j - mb * MARK_ROWS;
        const uint4 *mp = ix.marks + (size_t)mb * 4;
        uint4 q0 = __ldg(mp), q1 = __ldg(mp + 1), q2 = __ldg(mp + 2), q3 = __ldg(mp + 3);
        uint32_t w[16] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w,
                          q2.x, q2.y, q2.z, q2.w, q3.x, q3.y, q3.z, q3.w};
        uint32_t wi = mo >> 5, bi = mo & 31;
        uint32_t word = 0, before = 0;
#pragma unroll
        for (int x = 0; x < 15; x++) {
            if ((uint32_t)x < wi) before += __popc(w[1 + x]);
            if ((uint32_t)x == wi) word = w[1 + x];
        }
        if ((word >> bi) & 1u) {
            uint32_t rank = w[0] + before + __popc(word & ((1u << bi) - 1u));
            steps += t;
            return __ldg(ix.samples + rank) + t;
        }
        // LF step: c = BWT[j] (never $: the $ row has SA = 0, which is marked)
        uint32_t b = j / OCC_ROWS, o = j - b * OCC_ROWS;
        uint4 sup = __ldg(ix.super + b / SB_BLOCKS);
        OccBlock k;
        load_block(ix, b, o + 1, k);
        uint32_t c = block_symbol(k, o);
        uint32_t occ[4];
        occ_from(ix, b, o, sup, k, occ);
        uint32_t oc = c == 0 ? occ[0] : c == 1 ? occ[1] : c == 2 ? occ[2] : occ[3];
        uint32_t Cc = c == 0 ? ix.C[0] : c == 1 ? ix.C[1] : c == 2 ? ix.C[2] : ix.C[3];
        j = Cc + oc;
        t++;
    }
}

namespace {

// What the finishing kernels share.
struct FinishArgs {
    IndexView ix;
    Interval *ivs;
    const uint64_t *iv_off;
    const uint64_t *total;
    uint64_t *hit_off;
    uint64_t *hits;              // packed: pos | strand << 32 | mm << 40
    uint64_t n, capacity;
    uint32_t cap;
    uint32_t *lists;             // reads for a warp each from the front, for a block each from the back
    uint32_t *huge;              // reads with more than BLOCK_HITS hits from the front, those of long lists from the back
    SearchCtl *ctl;
};

__device__ __forceinline__ uint64_t hit_key(uint64_t raw)
{
    return ((raw & 0xffffffffull) << 1) | ((raw >> 32) & 1ull);   // (pos, strand)
}

// The hit of row (or, with IV_POS, position) x of an interval; without the
// suffix array its position is still the row (locate_hits).
__device__ __forceinline__ uint64_t hit_of(const IndexView &ix, uint32_t x, uint32_t meta)
{
    const uint32_t pos = (meta & IV_POS) || !ix.sa_ctx ? x : __ldg(&ix.sa_ctx[x].x);
    return (uint64_t)pos | ((uint64_t)((meta >> 2) & 1u) << 32) | ((uint64_t)(meta & 3u) << 40);
}

// Without the suffix array: the positions of a read's rows h[0, cnt), every
// nt-th by this thread (walks of up to s - 1 steps, so that all threads of the
// warp or block take part whatever the intervals' sizes).
__device__ __forceinline__ void locate_hits(const IndexView &ix, uint64_t *h, uint64_t cnt, uint32_t tid, uint32_t nt,
                                            uint32_t &steps)
{
    for (uint64_t i = tid; i < cnt; i += nt)
        h[i] = (h[i] & ~0xffffffffull) | locate_row(ix, (uint32_t)h[i], steps);
}

__device__ __forceinline__ void count_steps(SearchCtl *ctl, uint32_t steps)
{
    const unsigned mask = __activemask();
    const unsigned s = __reduce_add_sync(mask, steps);
    if (s && (threadIdx.x & 31) == (unsigned)(__ffs(mask) - 1)) atomicAdd(&ctl->lf_steps, (unsigned long long)s);
}

// Offsets of the listed hits; reads with at most SMALL_HITS of them, none cut
// off by the cap, are finished by their thread (an insertion into the hits
// it has written so far); the others go on a list.
__global__ void __launch_bounds__(TILE_THREADS) k_finish_small(const FinishArgs a, const uint64_t *__restrict__ sums,
                                                               bool scanned)
{
    __shared__ uint64_t ws[TILE_THREADS / 32];
    if (search_open(a.ctl)) return;
    uint64_t at = scanned ? sums[blockIdx.x] : tiles_before(sums, blockIdx.x, ws);
    uint32_t steps = 0;
    for (uint32_t i0 = 0; i0 < TILE; i0 += TILE_THREADS) {
        const uint64_t r = blockIdx.x * (uint64_t)TILE + i0 + threadIdx.x;
        const uint64_t t = r < a.n ? a.total[r] : 0;
        const uint64_t keep = a.cap && t > a.cap ? a.cap : t;
        uint64_t all;
        const uint64_t q0 = at + block_exclusive(keep, ws, all);
        at += all;
        if (r < a.n) a.hit_off[r] = q0;
        if (r + 1 == a.n || (a.n == 0 && r == 0)) {
            a.hit_off[a.n] = q0 + keep;
            a.ctl->post_hits = q0 + keep;
        }
        if (keep == 0 || q0 + keep > a.capacity) continue;
        const uint64_t b = a.iv_off[r], e = a.iv_off[r + 1];
        // (without the suffix array a hit is a walk: more than one goes to a warp's lanes)
        if (keep > (a.ix.sa_ctx ? SMALL_HITS : 1u) || t > keep || e - b > 32) {
            if (keep > BLOCK_HITS) a.huge[atomicAdd(&a.ctl->n_huge, 1u)] = (uint32_t)r;
            else if (e - b > LONG_LIST) a.huge[a.n - 1 - atomicAdd(&a.ctl->n_long, 1u)] = (uint32_t)r;
            else if (keep <= WARP_HITS && e - b <= WARP_HITS && (t == keep || a.cap <= WARP_CAP))
                a.lists[atomicAdd(&a.ctl->n_warp, 1u)] = (uint32_t)r;
            else a.lists[a.n - 1 - atomicAdd(&a.ctl->n_block, 1u)] = (uint32_t)r;
            continue;
        }
        uint64_t q = q0;
        for (uint64_t x = b; x < e; x++) {
            const Interval v = a.ivs[x];
            for (uint32_t row = v.l; row < v.r; row++, q++) {
                uint64_t h = hit_of(a.ix, row, v.meta);
                if (!a.ix.sa_ctx) locate_hits(a.ix, &h, 1, 0, 1, steps);
                const uint64_t kh = hit_key(h);
                uint64_t w = q;
                for (; w > q0; w--) {
                    const uint64_t p = a.hits[w - 1];
                    if (hit_key(p) < kh) break;
                    a.hits[w] = p;
                }
                a.hits[w] = h;
            }
        }
    }
    if (!a.ix.sa_ctx) count_steps(a.ctl, steps);
}

// Bitonic sort of the packed hits sh[0, P) (P a power of two, padding ~0 last)
// by (pos, strand), by the `nt` threads numbered `tid` of a warp (BLOCK false)
// or a block (true), which meet at a barrier between phases: log2(P) (log2(P)
// + 1) / 2 phases, each thread taking every nt-th compare-exchange pair
// (i, i ^ jj) with i's jj bit clear (the pairs of a phase are disjoint); a
// thread loads up to four pairs before it compares and stores any of them.
template <bool BLOCK>
__device__ __forceinline__ void bitonic_hits(uint64_t *sh, uint32_t P, uint32_t tid, uint32_t nt)
{
    for (uint32_t kk = 2; kk <= P; kk <<= 1)
        for (uint32_t jj = kk >> 1; jj > 0; jj >>= 1) {
            for (uint32_t t0 = tid; t0 < P / 2; t0 += 4 * nt) {
                uint32_t ii[4];
                uint64_t xs[4], ys[4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const uint32_t t = t0 + (uint32_t)u * nt;
                    ii[u] = ((t & ~(jj - 1)) << 1) | (t & (jj - 1));
                    if (t < P / 2) { xs[u] = sh[ii[u]]; ys[u] = sh[ii[u] ^ jj]; }
                }
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const uint32_t t = t0 + (uint32_t)u * nt;
                    if (t < P / 2) {
                        const uint64_t kx = xs[u] == ~0ull ? ~0ull : hit_key(xs[u]);
                        const uint64_t ky = ys[u] == ~0ull ? ~0ull : hit_key(ys[u]);
                        if ((kx > ky) == ((ii[u] & kk) == 0)) { sh[ii[u]] = ys[u]; sh[ii[u] ^ jj] = xs[u]; }
                    }
                }
            }
            if (BLOCK) __syncthreads(); else __syncwarp();
        }
}

// The packed hits sh[0, cnt) of one read to out[0, cnt), sorted by (pos,
// strand), by the `nt` threads `tid` of a warp or a block.  Hits within `span`
// positions of each other (those of a tandem array) are ordered by counting:
// a bit per (position, strand) from the first one (no two hits share one), a
// prefix sum over the words' bit counts, and each hit goes to the number of
// bits below its own; else a bitonic sort, for which sh holds a power of two
// of entries.
template <bool BLOCK>
__device__ __forceinline__ void sort_hits(uint64_t *sh, uint32_t cnt, uint32_t *bits, uint32_t *pre, uint32_t span,
                                          uint64_t *__restrict__ out, uint32_t tid, uint32_t nt)
{
    __shared__ uint32_t red[2][LONG_THREADS / 32];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t lo = 0xffffffffu, hi = 0;
    for (uint32_t i = tid; i < cnt; i += nt) {
        const uint32_t p = (uint32_t)sh[i];
        lo = min(lo, p);
        hi = max(hi, p);
    }
    lo = __reduce_min_sync(FULL, lo);
    hi = __reduce_max_sync(FULL, hi);
    if (BLOCK) {
        if (lane == 0) { red[0][warp] = lo; red[1][warp] = hi; }
        __syncthreads();
        for (uint32_t w = 0; w < nt / 32; w++) { lo = min(lo, red[0][w]); hi = max(hi, red[1][w]); }
        __syncthreads();
    }
    if (hi - lo < span) {
        const uint32_t words = (hi - lo) / 16u + 1u, per = (words + nt - 1) / nt;
        for (uint32_t i = tid; i < words; i += nt) bits[i] = 0;
        if (BLOCK) __syncthreads(); else __syncwarp();
        for (uint32_t i = tid; i < cnt; i += nt) {
            const uint32_t k = 2u * ((uint32_t)sh[i] - lo) + (uint32_t)((sh[i] >> 32) & 1u);
            atomicOr(&bits[k >> 5], 1u << (k & 31u));
        }
        if (BLOCK) __syncthreads(); else __syncwarp();
        uint32_t sum = 0;
        for (uint32_t i = tid * per; i < min(words, (tid + 1) * per); i++) sum += __popc(bits[i]);
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, incl, o);
            if ((int)lane >= o) incl += y;
        }
        uint32_t base = incl - sum;
        if (BLOCK) {
            if (lane == 31) red[0][warp] = incl;
            __syncthreads();
            for (uint32_t w = 0; w < warp; w++) base += red[0][w];
        }
        for (uint32_t i = tid * per; i < min(words, (tid + 1) * per); i++) { pre[i] = base; base += __popc(bits[i]); }
        if (BLOCK) __syncthreads(); else __syncwarp();
        for (uint32_t i = tid; i < cnt; i += nt) {
            const uint64_t h = sh[i];
            const uint32_t k = 2u * ((uint32_t)h - lo) + (uint32_t)((h >> 32) & 1u);
            out[pre[k >> 5] + __popc(bits[k >> 5] & ((1u << (k & 31u)) - 1u))] = h;
        }
        return;
    }
    uint32_t P = 1;
    while (P < cnt) P <<= 1;
    for (uint32_t i = cnt + tid; i < P; i += nt) sh[i] = ~0ull;
    if (BLOCK) __syncthreads(); else __syncwarp();
    bitonic_hits<BLOCK>(sh, P, tid, nt);
    for (uint32_t i = tid; i < cnt; i += nt) out[i] = sh[i];
}

// Where a block cuts a read's list of intervals ivs[b, e) with more than cap
// rows: the first cap rows in the order (d, strand, row) are the intervals of
// the classes (d, strand) before `cls`, those of cls whose row is below `row`,
// and the first `take` rows of cls's interval at `row`.
struct Cut {
    uint32_t cls, row, take;
};

__device__ __forceinline__ uint32_t iv_class(const Interval &x) { return ((x.meta & 3u) << 1) | ((x.meta >> 2) & 1u); }

// The rows per class come first (no row is looked up for that); then the class
// that crosses the cap is searched by its rows, eight bits a pass: a pass sums
// the rows under each of the 256 next values.
template <uint32_t NT>
__device__ __forceinline__ Cut find_cut(Interval *ivs, uint64_t b, uint64_t e, uint32_t cap,
                                        const uint32_t *__restrict__ isa, unsigned long long *hist, uint32_t *found)
{
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    uint64_t in_class[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (uint64_t i = b + tid; i < e; i += NT) {
        const Interval x = ivs[i];
        const uint32_t c = iv_class(x), z = x.r - x.l;
#pragma unroll
        for (uint32_t q = 0; q < 8; q++) in_class[q] += c == q ? z : 0u;
    }
    if (tid < 8) hist[tid] = 0;
    __syncthreads();
#pragma unroll
    for (uint32_t q = 0; q < 8; q++) {
        uint64_t v = in_class[q];
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
        if (lane == 0 && v) atomicAdd(&hist[q], (unsigned long long)v);
    }
    __syncthreads();
    Cut c{0, 0, 0};
    uint64_t before = 0;
    while (before + hist[c.cls] < cap) before += hist[c.cls++];
    __syncthreads();
    for (int sh = 24; sh >= 0; sh -= 8) {
        for (uint32_t i = tid; i < 256; i += NT) hist[i] = 0;
        __syncthreads();
        for (uint64_t i = b + tid; i < e; i += NT) {
            Interval x = ivs[i];
            if (iv_class(x) != c.cls || x.r <= x.l) continue;
            if (sh == 24 && (x.meta & IV_POS)) {
                to_rows(x, isa);
                ivs[i] = x;   // (the passes keep this stride)
            }
            if (((uint64_t)x.l >> (sh + 8)) == ((uint64_t)c.row >> (sh + 8)))
                atomicAdd(&hist[(x.l >> sh) & 255u], (unsigned long long)(x.r - x.l));
        }
        __syncthreads();
        if (tid < 32) {
            uint64_t part[8], sum = 0;
#pragma unroll
            for (int i = 0; i < 8; i++) { part[i] = hist[lane * 8 + i]; sum += part[i]; }
            uint64_t incl = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint64_t y = __shfl_up_sync(FULL, incl, o);
                if ((int)lane >= o) incl += y;
            }
            uint64_t run = before + incl - sum;   // rows before this lane's values
            // the first value with which the rows counted reach the cap
            int digit = -1;
            uint64_t rows = 0;
#pragma unroll
            for (int i = 0; i < 8; i++) {
                if (digit < 0 && run + part[i] >= cap) { digit = (int)lane * 8 + i; rows = run; }
                run += part[i];
            }
            const unsigned has = __ballot_sync(FULL, digit >= 0);
            if ((int)lane == __ffs(has) - 1) { found[0] = (uint32_t)digit; found[1] = (uint32_t)rows; }
        }
        __syncthreads();
        c.row |= found[0] << sh;
        before = found[1];   // (less than cap)
        __syncthreads();
    }
    c.take = cap - (uint32_t)before;
    return c;
}

// The read's listed rows as hits to out[0, ...), in no order, by a block: all
// rows of its intervals, or those the cut keeps.  count: in shared memory.
template <uint32_t NT>
__device__ __forceinline__ void expand_block(const IndexView &ix, const Interval *ivs, uint64_t b, uint64_t e, bool over,
                                             const Cut &c, uint64_t *out, unsigned long long *count)
{
    const uint32_t lane = threadIdx.x & 31;
    if (threadIdx.x == 0) *count = 0;
    __syncthreads();
    for (uint64_t c0 = b + (threadIdx.x & ~31u); c0 < e; c0 += NT) {
        Interval x{};
        if (c0 + lane < e) x = ivs[c0 + lane];
        uint32_t sz = x.r - x.l;
        if (over && sz) {
            const uint32_t k = iv_class(x);
            if (k > c.cls || (k == c.cls && x.l > c.row)) sz = 0;
            else if (k == c.cls && x.l == c.row) sz = c.take;
        }
        uint32_t incl = sz;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, incl, o);
            if ((int)lane >= o) incl += y;
        }
        unsigned long long at = 0;
        if (lane == 31 && incl) at = atomicAdd(count, (unsigned long long)incl);
        at = __shfl_sync(FULL, at, 31) + incl - sz;
        if (sz == 1) out[at] = hit_of(ix, x.l, x.meta);
        for (unsigned todo = __ballot_sync(FULL, sz > 1); todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const uint32_t wl = __shfl_sync(FULL, x.l, src), wz = __shfl_sync(FULL, sz, src);
            const uint32_t wm = __shfl_sync(FULL, x.meta, src);
            const unsigned long long wa = __shfl_sync(FULL, at, src);
            for (uint32_t i = lane; i < wz; i += 32) out[wa + i] = hit_of(ix, wl + i, wm);
        }
    }
    __syncthreads();
}

// A warp's intervals, S of them a lane at most: the key K at which the rows
// counted in key order reach keep, and the rows before it.  Keys are distinct,
// so a bitwise search from the top bit finds it.
template <uint32_t S>
__device__ __forceinline__ void cut_key(const uint64_t *key, const uint32_t *sz, uint32_t keep, uint64_t &prefix,
                                        uint32_t &before)
{
    prefix = 0;
    before = 0;
    for (int bit = 34; bit >= 0; bit--) {
        const uint64_t hi = prefix >> (bit + 1);
        uint32_t z = 0;
#pragma unroll
        for (uint32_t i = 0; i < S; i++)
            if ((key[i] >> (bit + 1)) == hi && !((key[i] >> bit) & 1u)) z += sz[i];
        z = __reduce_add_sync(FULL, z);
        if (before + z < keep) { before += z; prefix |= 1ull << bit; }
    }
}

// Reads of up to WARP_HITS hits and intervals: one warp each, taken from the
// list by a counter (reads differ a lot in size: a fixed stride left one warp
// with the largest).  Each lane holds up to eight intervals in registers.
// (The cut of a read over its cap goes through one, two or all eight, and a
// single interval needs none.  It was bound by instructions: 100k reads over a
// cap of 10 took 0.61 ms here whether they had one interval or 50, now 0.19 and
// 0.31.)
// sh, bits, pre: the warp's own shared memory.
__device__ __forceinline__ void finish_by_warps(const FinishArgs &a, uint64_t *sh, uint32_t *bits, uint32_t *pre,
                                                uint32_t &steps)
{
    const uint32_t lane = threadIdx.x & 31;
    const unsigned n_list = a.ctl->n_warp;
    constexpr uint32_t PER = WARP_HITS / 32;
    for (;;) {
        unsigned bi = 0;
        if (lane == 0) bi = atomicAdd(&a.ctl->next_warp, 1u);
        bi = __shfl_sync(FULL, bi, 0);
        if (bi >= n_list) break;
        const uint32_t r = a.lists[bi];
        const uint64_t b = a.iv_off[r], q0 = a.hit_off[r], t = a.total[r];
        const uint32_t ni = (uint32_t)(a.iv_off[r + 1] - b), keep = (uint32_t)(a.hit_off[r + 1] - q0);
        uint32_t l[PER], sz[PER], meta[PER];
#pragma unroll
        for (uint32_t i = 0; i < PER; i++) {
            const uint32_t x = i * 32 + lane;
            l[i] = sz[i] = meta[i] = 0;
            if (x < ni) {
                const Interval v = a.ivs[b + x];
                l[i] = v.l; sz[i] = v.r - v.l; meta[i] = v.meta;
            }
        }
        if (t > keep) {
            // over the cap: the first keep rows in the order (d, strand, row) (sizes cut at 2^16,
            // more than any cap taken here)
            uint64_t key[PER];
#pragma unroll
            for (uint32_t i = 0; i < PER; i++) {
                Interval v;
                v.l = l[i]; v.r = l[i] + sz[i]; v.meta = meta[i]; v.read = r;
                if (sz[i]) to_rows(v, a.ix.isa);
                l[i] = v.l; meta[i] = v.meta;
                key[i] = iv_key(v);
                if (sz[i] == 0) key[i] = ~0ull;
                sz[i] = min(sz[i], WARP_CAP + 1u);
            }
            uint64_t prefix = __shfl_sync(FULL, key[0], 0);   // (of a single interval)
            uint32_t before = 0;
            if (ni > 64) cut_key<PER>(key, sz, keep, prefix, before);
            else if (ni > 32) cut_key<2>(key, sz, keep, prefix, before);
            else if (ni > 1) cut_key<1>(key, sz, keep, prefix, before);
#pragma unroll
            for (uint32_t i = 0; i < PER; i++) {
                if (key[i] == prefix) sz[i] = keep - before;
                else if (key[i] > prefix) sz[i] = 0;
            }
        }
        // the rows' hits, lane by lane; an interval of several rows by the whole warp
        uint32_t mine = 0;
#pragma unroll
        for (uint32_t i = 0; i < PER; i++) mine += sz[i];
        uint32_t at = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, at, o);
            if ((int)lane >= o) at += y;
        }
        at -= mine;
#pragma unroll
        for (uint32_t i = 0; i < PER; i++) {
            if (i * 32u >= ni) break;
            if (sz[i] == 1) sh[at] = hit_of(a.ix, l[i], meta[i]);
            for (unsigned todo = __ballot_sync(FULL, sz[i] > 1); todo; todo &= todo - 1) {
                const int src = __ffs(todo) - 1;
                const uint32_t wl = __shfl_sync(FULL, l[i], src), wz = __shfl_sync(FULL, sz[i], src);
                const uint32_t wm = __shfl_sync(FULL, meta[i], src), wa = __shfl_sync(FULL, at, src);
                for (uint32_t x = lane; x < wz; x += 32) sh[wa + x] = hit_of(a.ix, wl + x, wm);
            }
            at += sz[i];
        }
        __syncwarp();
        if (!a.ix.sa_ctx) {
            locate_hits(a.ix, sh, keep, lane, 32, steps);
            __syncwarp();
        }
        sort_hits<false>(sh, keep, bits, pre, WARP_SPAN, a.hits + q0, lane, 32);
        __syncwarp();
    }
}

// Larger reads (up to BLOCK_HITS hits): one block each, taken by a counter;
// then, in the small blocks, a warp each for the others (the largest first: a
// kernel for each kind had every kind's last reads run alone).
// Those with the longest lists (a read in a diverged tandem array has 10^5
// intervals of a row each) have blocks of 1,024 threads: 128 took 0.65 ms
// for the longest of a million reads.
template <uint32_t NT>
__global__ void __launch_bounds__(NT) k_finish_block(const FinishArgs a)
{
    __shared__ uint64_t sh[BLOCK_HITS];
    __shared__ uint32_t bits[BLOCK_SPAN / 16], pre[BLOCK_SPAN / 16];
    __shared__ unsigned long long count;
    __shared__ uint32_t found[2];
    __shared__ unsigned bi_s;
    if (search_open(a.ctl)) return;
    constexpr bool LONG = NT == LONG_THREADS;
    const unsigned n_list = LONG ? a.ctl->n_long : a.ctl->n_block;
    uint32_t steps = 0;
    for (;;) {
        if (threadIdx.x == 0) bi_s = atomicAdd(LONG ? &a.ctl->next_long : &a.ctl->next_block, 1u);
        __syncthreads();
        const unsigned bi = bi_s;
        __syncthreads();
        if (bi >= n_list) break;
        const uint32_t r = (LONG ? a.huge : a.lists)[a.n - 1 - bi];
        const uint64_t b = a.iv_off[r], e = a.iv_off[r + 1], q0 = a.hit_off[r];
        const uint32_t keep = (uint32_t)(a.hit_off[r + 1] - q0);
        const bool over = a.total[r] > keep;
        Cut c{0, 0, 0};
        if (over) c = find_cut<NT>(a.ivs, b, e, a.cap, a.ix.isa, (unsigned long long *)sh, found);
        expand_block<NT>(a.ix, a.ivs, b, e, over, c, sh, &count);
        if (!a.ix.sa_ctx) {
            locate_hits(a.ix, sh, keep, threadIdx.x, NT, steps);
            __syncthreads();
        }
        sort_hits<true>(sh, keep, bits, pre, BLOCK_SPAN, a.hits + q0, threadIdx.x, NT);
        __syncthreads();
    }
    if (!LONG) {
        const uint32_t wi = threadIdx.x >> 5;
        static_assert(WARP_HITS * (BLOCK_READ_THREADS / 32) <= BLOCK_HITS &&
                      WARP_SPAN * (BLOCK_READ_THREADS / 32) <= BLOCK_SPAN, "the warps' shares of the block's arrays");
        finish_by_warps(a, sh + wi * WARP_HITS, bits + wi * (WARP_SPAN / 16), pre + wi * (WARP_SPAN / 16), steps);
    }
    if (!a.ix.sa_ctx) count_steps(a.ctl, steps);
}

// Reads above BLOCK_HITS hits (only without a cap or with a cap above it): a
// block each writes the hits, not yet in order.
__global__ void __launch_bounds__(LONG_THREADS) k_finish_huge(const FinishArgs a, uint32_t n_huge)
{
    __shared__ unsigned long long hist[256], count;
    __shared__ uint32_t found[2];
    uint32_t steps = 0;
    for (uint32_t i = blockIdx.x; i < n_huge; i += gridDim.x) {
        const uint32_t r = a.huge[i];
        const uint64_t b = a.iv_off[r], e = a.iv_off[r + 1], q0 = a.hit_off[r];
        const bool over = a.total[r] > a.hit_off[r + 1] - q0;
        Cut c{0, 0, 0};
        if (over) c = find_cut<LONG_THREADS>(a.ivs, b, e, a.cap, a.ix.isa, hist, found);
        expand_block<LONG_THREADS>(a.ix, a.ivs, b, e, over, c, a.hits + q0, &count);
        if (!a.ix.sa_ctx) locate_hits(a.ix, a.hits + q0, count, threadIdx.x, LONG_THREADS, steps);
        __syncthreads();
    }
    if (!a.ix.sa_ctx) count_steps(a.ctl, steps);
}

// one read with more than BLOCK_HITS hits: bitonic network over a global scratch
__global__ void __launch_bounds__(1024) k_sort_global(uint64_t *__restrict__ hits, uint64_t cnt,
                                                      uint64_t *__restrict__ scratch, uint64_t P)
{
    for (uint64_t i = threadIdx.x; i < P; i += blockDim.x) scratch[i] = i < cnt ? hits[i] : ~0ull;
    __syncthreads();
    for (uint64_t kk = 2; kk <= P; kk <<= 1)
        for (uint64_t jj = kk >> 1; jj > 0; jj >>= 1) {
            for (uint64_t i = threadIdx.x; i < P; i += blockDim.x) {
                uint64_t p = i ^ jj;
                if (p > i) {
                    uint64_t x = scratch[i], y = scratch[p];
                    bool up = (i & kk) == 0;
                    uint64_t kx = x == ~0ull ? ~0ull : hit_key(x), ky = y == ~0ull ? ~0ull : hit_key(y);
                    if ((kx > ky) == up) { scratch[i] = y; scratch[p] = x; }
                }
            }
            __syncthreads();
        }
    for (uint64_t i = threadIdx.x; i < cnt; i += blockDim.x) hits[i] = scratch[i];
}

__global__ void k_debug_occ(const IndexView ix, const uint64_t *__restrict__ rows, uint64_t n,
                            uint32_t *__restrict__ out)
{
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t j = (uint32_t)rows[i];
        uint32_t ol[4], orr[4];
        occ_pair(ix, j, j, ol, orr);
        for (int c = 0; c < 4; c++) out[4 * i + c] = ol[c];
    }
}

__global__ void k_debug_locate(const IndexView ix, const uint64_t *__restrict__ rows, uint64_t n,
                               uint32_t *__restrict__ out)
{
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t steps = 0;
        out[i] = locate_row(ix, (uint32_t)rows[i], steps);
    }
}

__global__ void k_debug_seed(const IndexView ix, const uint32_t *__restrict__ codes, uint32_t len, uint64_t n,
                             uint32_t *__restrict__ out)
{
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t l, r;
        seed_interval(ix, codes[i], len, l, r);
        out[2 * i] = l;
        out[2 * i + 1] = r < l ? l : r;
    }
}

unsigned grid1(uint64_t n, int block = 256)
{
    return (unsigned)std::min<uint64_t>(std::max<uint64_t>((n + block - 1) / block, 1), 152ull * 64);
}

}  // namespace

// Exclusive scan of n uint64 counts into n + 1 offsets with caller-provided
// tile scratch of at least n / 2048 + 2 entries (no allocation).
int exclusive_scan_u64_scratch(const uint64_t *in, uint64_t n, uint64_t *out, unsigned long long *scratch,
                               cudaStream_t s)
{
    uint64_t ntiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    uint64_t *ts = (uint64_t *)scratch;
    if (ntiles) k_scan_tiles<uint64_t><<<(unsigned)ntiles, SCAN_THREADS, 0, s>>>(in, n, out, ts);
    k_scan_sums<<<1, 1024, 0, s>>>(ts, ntiles);
    unsigned g = (unsigned)std::min<uint64_t>(std::max<uint64_t>((n + 255) / 256, 1), 152 * 32);
    k_scan_add<<<g, 256, 0, s>>>(out, n, ts);
    MICA_CUDA_TRY(cudaGetLastError());
    return 0;
}

static uint64_t big_list_bytes(uint64_t n)
{
    return (std::max<uint64_t>(n, 1) * 4 + 15) & ~15ull;
}

// w.big holds the list of reads for warps and blocks of their own (a read
// is on one of them: n u32), then the list of larger ones (n u32); w.scan_tmp
// the tile sums of the interval counts, then of the listed hits.
static uint64_t post_list_bytes(uint64_t n) { return 2 * big_list_bytes(n); }
static uint64_t tiles_of(uint64_t n) { return std::max<uint64_t>(1, (n + TILE - 1) / TILE); }
static uint64_t tile_bytes(uint64_t n) { return (2 * tiles_of(n) + 1) * 8; }

static FinishArgs finish_args(const mica_index *idx, Workspace &w, uint64_t n, uint32_t hit_cap, uint64_t capacity)
{
    FinishArgs a;
    a.ix = idx->view;
    a.ivs = (Interval *)w.iv_sorted.p;
    a.iv_off = (const uint64_t *)w.iv_off.p;
    a.total = (const uint64_t *)w.total.p;
    a.hit_off = (uint64_t *)w.hit_off.p;
    a.hits = (uint64_t *)w.hits.p;
    a.n = n;
    a.capacity = capacity;
    a.cap = hit_cap;
    a.lists = (uint32_t *)w.big.p;
    a.huge = (uint32_t *)((char *)w.big.p + big_list_bytes(n));
    a.ctl = (SearchCtl *)w.ctl.p;
    return a;
}

// Steps 1 to 3: intervals grouped by read, totals, tile sums of the listed hits.
static int enqueue_totals(Workspace &w, uint64_t n, uint32_t hit_cap, uint32_t report, bool need_total,
                          cudaStream_t s, uint64_t &L)
{
    uint64_t *iv_off = (uint64_t *)w.iv_off.p, *sums = (uint64_t *)w.scan_tmp.p;
    SearchCtl *ctl = (SearchCtl *)w.ctl.p;
    const unsigned tiles = (unsigned)tiles_of(n);
    if (tiles > 1) {
        k_tile_counts<<<tiles, TILE_THREADS, 0, s>>>((const uint32_t *)w.iv_cnt.p, n, sums);
        L++;
    }
    if (tiles > SCAN_TILES) {
        k_scan_sums<<<1, 1024, 0, s>>>(sums, tiles);
        L++;
    }
    unsigned long long *total = (unsigned long long *)w.total.p;
    k_offsets<<<tiles, TILE_THREADS, 0, s>>>((const uint32_t *)w.iv_cnt.p, n, sums, tiles > SCAN_TILES, iv_off,
                                             (uint64_t *)total);
    const unsigned g = (unsigned)std::min<uint64_t>(152 * 16, std::max<uint64_t>(8, n / 64));
    k_iv_scatter<<<g, 256, 0, s>>>((const Interval *)w.iv.p, ctl, w.iv_cap, iv_off, (uint32_t *)w.iv_cnt.p,
                                   (Interval *)w.iv_sorted.p, total);
    if (report == MICA_REPORT_BEST_STRATUM) {
        k_stratum<<<grid1(n, 128), 128, 0, s>>>((Interval *)w.iv_sorted.p, iv_off, n, (uint64_t *)total, ctl);
        L++;
    }
    if (tiles > 1 || need_total) {   // (a single tile has none before it)
        k_listed<<<tiles, TILE_THREADS, 0, s>>>((const uint64_t *)total, n, hit_cap, sums + tiles);
        L++;
    }
    if (tiles > SCAN_TILES) {
        k_scan_sums<<<1, 1024, 0, s>>>(sums + tiles, tiles);
        L++;
    }
    L += 2;
    MICA_CUDA_TRY(cudaGetLastError());
    return 0;
}

// Steps 4 and 5.
static int enqueue_finish(const FinishArgs &a, Workspace &w, cudaStream_t s, uint64_t &L)
{
    const unsigned tiles = (unsigned)tiles_of(a.n);
    k_finish_small<<<tiles, TILE_THREADS, 0, s>>>(a, (const uint64_t *)w.scan_tmp.p + tiles, tiles > SCAN_TILES);
    const uint64_t n1 = std::max<uint64_t>(a.n, 1);
    k_finish_block<LONG_THREADS><<<(unsigned)std::min<uint64_t>(152, n1), LONG_THREADS, 0, s>>>(a);
    k_finish_block<BLOCK_READ_THREADS><<<(unsigned)std::min<uint64_t>(152 * 5, n1), BLOCK_READ_THREADS, 0, s>>>(a);
    L += 3;
    MICA_CUDA_TRY(cudaGetLastError());
    return 0;
}

// The whole post-search pipeline for one batch, enqueued with every count
// read on the device (fixed grids, capacity-guarded writes) so it can be
// captured in a CUDA graph.  Buffers must already hold `hit_capacity` hits.
// Ends with a copy of the control block (the search's counters, the hit
// total, locate steps and list counts) into pinned host memory `status`.
int enqueue_post_device(const mica_index *idx, Workspace &w, const ReadsView &rd, uint32_t hit_cap,
                        uint32_t report, uint64_t hit_capacity, cudaStream_t s, void *status, uint64_t &L)
{
    if (int rc = enqueue_totals(w, rd.n, hit_cap, report, false, s, L)) return rc;
    if (int rc = enqueue_finish(finish_args(idx, w, rd.n, hit_cap, hit_capacity), w, s, L)) return rc;
    MICA_CUDA_TRY(cudaMemcpyAsync(status, w.ctl.p, sizeof(SearchCtl), cudaMemcpyDeviceToHost, s));
    return 0;
}

// Reserve every post-search buffer for n reads and hit_capacity hits.
// Device bytes reserve_post takes for n reads (the sizes below).
uint64_t post_workspace_bytes(uint64_t n, uint64_t iv_cap, uint64_t hit_capacity)
{
    return std::max<uint64_t>(iv_cap, 1) * sizeof(Interval) + 2 * (n + 1) * 8 + std::max<uint64_t>(n, 1) * 8 +
           post_list_bytes(n) + tile_bytes(n) + std::max<uint64_t>(hit_capacity, 1) * sizeof(Hit) + 64;
}

int reserve_post(Workspace &w, uint64_t n, uint32_t iv_cap, uint64_t hit_capacity)
{
    int rc;
    if ((rc = dev_reserve(w.iv_sorted, std::max<uint64_t>(iv_cap, 1) * sizeof(Interval))) ||
        (rc = dev_reserve(w.iv_off, (n + 1) * 8)) || (rc = dev_reserve(w.total, std::max<uint64_t>(n, 1) * 8)) ||
        (rc = dev_reserve(w.hit_off, (n + 1) * 8)) || (rc = dev_reserve(w.big, post_list_bytes(n))) ||
        (rc = dev_reserve(w.scan_tmp, tile_bytes(n))) ||
        (rc = dev_reserve(w.hits, std::max<uint64_t>(hit_capacity, 1) * sizeof(Hit) + 64)))
        return rc;
    return 0;
}

int run_post(const mica_index *idx, Workspace &w, mica_stats &stt, const ReadsView &rd, uint32_t hit_cap,
             uint32_t report, cudaStream_t s, uint64_t *n_hits_out)
{
    const uint64_t n = rd.n;
    int rc;
    if ((rc = reserve_post(w, n, (uint32_t)stt.intervals, 1))) return rc;
    uint64_t &L = stt.launches;
    SearchCtl *ctl = (SearchCtl *)w.ctl.p;
    // the control block's post-search fields (a search may have run in several launches)
    MICA_CUDA_TRY(cudaMemsetAsync(&ctl->post_hits, 0, sizeof(SearchCtl) - offsetof(SearchCtl, post_hits), s));
    if ((rc = enqueue_totals(w, n, hit_cap, report, true, s, L))) return rc;
    const unsigned tiles = (unsigned)tiles_of(n);
    uint64_t *sums = (uint64_t *)w.scan_tmp.p;
    if (tiles <= SCAN_TILES) {   // (the scan leaves it there)
        k_tiles_total<<<1, TILE_THREADS, 0, s>>>(sums + tiles, tiles, sums + 2 * tiles);
        L++;
    }
    uint64_t nh = 0;
    MICA_CUDA_TRY(cudaMemcpyAsync(&nh, sums + 2 * tiles, 8, cudaMemcpyDeviceToHost, s));
    MICA_CUDA_TRY(cudaStreamSynchronize(s));
    if ((rc = dev_reserve(w.hits, std::max<uint64_t>(nh, 1) * sizeof(Hit) + 64))) return rc;
    const FinishArgs a = finish_args(idx, w, n, hit_cap, nh);
    if ((rc = enqueue_finish(a, w, s, L))) return rc;
    SearchCtl out;
    MICA_CUDA_TRY(cudaMemcpyAsync(&out, ctl, sizeof(out), cudaMemcpyDeviceToHost, s));
    MICA_CUDA_TRY(cudaStreamSynchronize(s));
    if (out.n_huge) {
        k_finish_huge<<<std::min(out.n_huge, 152u), LONG_THREADS, 0, s>>>(a, out.n_huge);
        L++;
        std::vector<uint32_t> huge(out.n_huge);
        MICA_CUDA_TRY(cudaMemcpyAsync(huge.data(), a.huge, 4ull * out.n_huge, cudaMemcpyDeviceToHost, s));
        MICA_CUDA_TRY(cudaMemcpyAsync(&out, ctl, sizeof(out), cudaMemcpyDeviceToHost, s));
        MICA_CUDA_TRY(cudaStreamSynchronize(s));
        for (uint32_t r : huge) {
            uint64_t ob[2];
            MICA_CUDA_TRY(cudaMemcpy(ob, a.hit_off + r, 16, cudaMemcpyDeviceToHost));
            uint64_t cnt = ob[1] - ob[0];
            uint64_t P = 1;
            while (P < cnt) P <<= 1;
            DevBuf scratch;
            if ((rc = dev_reserve(scratch, P * 8))) return rc;
            k_sort_global<<<1, 1024, 0, s>>>((uint64_t *)w.hits.p + ob[0], cnt, (uint64_t *)scratch.p, P);
            L++;
            MICA_CUDA_TRY(cudaStreamSynchronize(s));
            dev_release(scratch);
        }
    }
    MICA_CUDA_TRY(cudaGetLastError());
    stt.located = nh;
    stt.lf_steps = out.lf_steps;
    *n_hits_out = nh;
    return 0;
}

int debug_occ(const mica_index *idx, const uint64_t *d_rows, uint64_t n, uint32_t *d_out, cudaStream_t s)
{
    if (n) k_debug_occ<<<grid1(n), 256, 0, s>>>(idx->view, d_rows, n, d_out);
    MICA_CUDA_TRY(cudaGetLastError());
    return 0;
}

int debug_seed(const mica_index *idx, const uint32_t *d_codes, uint32_t len, uint64_t n, uint32_t *d_out,
               cudaStream_t s)
{
    if (n) k_debug_seed<<<grid1(n), 256, 0, s>>>(idx->view, d_codes, len, n, d_out);
    MICA_CUDA_TRY(cudaGetLastError());
    return 0;
}

int debug_locate(const mica_index *idx, const uint64_t *d_rows, uint64_t n, uint32_t *d_out, cudaStream_t s)
{
    if (n) k_debug_locate<<<grid1(n), 256, 0, s>>>(idx->view, d_rows, n, d_out);
    MICA_CUDA_TRY(cudaGetLastError());
    return 0;
}

}  // namespace mica

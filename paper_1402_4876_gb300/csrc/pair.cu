// Mate pairing of a paired-end batch (the paper reports properly paired
// reads, Section 3, Table 1): for pair i (reads 2i and 2i + 1), every listed
// + strand hit of one mate against every listed - strand hit of the other
// whose fragment length b.pos + m_b - a.pos lies in the insert window.
//
// A read's hits are sorted by (pos, strand), so for a + strand hit a the -
// strand partners form one contiguous position range of the other mate's list,
// which two binary searches find.  A pair with a few hits is one thread's.  The
// others go on a list, one warp each, taken by a counter: 32 + strand hits at
// a time look their ranges up, and the ranges' (a, b) combinations are dealt
// out evenly to the lanes, whose counts and best placements are merged at the
// end.
//
// What bounds it: two mates in one tandem array have up to cap hits each and
// some 10^5 combinations, the rest of a batch one or two.  One thread per
// pair took 5.4 ms for the 500k pairs of a 512 Mbp human-like genome, all but
// a fraction of it the longest pair's.
#include <algorithm>

#include "mica_internal.cuh"

namespace mica {
namespace {

struct Best {
    uint32_t n = 0, nbest = 0, mm = 0xffu, pp = 0, pm = 0, mate = 0;
};

// Offer combination (a = + strand hit of `amate`, b = - strand hit).
__device__ __forceinline__ void offer(Best &B, uint32_t mm, uint32_t pp, uint32_t amate, uint32_t pm)
{
    B.n = B.n == 0xffffffffu ? B.n : B.n + 1;
    bool better = mm < B.mm || (mm == B.mm && (pp < B.pp || (pp == B.pp && (amate < B.mate ||
                                                                              (amate == B.mate && pm < B.pm)))));
    if (mm < B.mm) B.nbest = 1;
    else if (mm == B.mm) B.nbest++;
    if (better) { B.mm = mm; B.pp = pp; B.pm = pm; B.mate = amate; }
}

constexpr unsigned PFULL = 0xffffffffu;
constexpr uint32_t PAIR_SMALL = 8;     // pairs with at most this many hits, both mates together: one thread each
constexpr uint64_t PAIR_LARGE = 1ull << 26;   // (a warp's 32-bit counts hold 32 ranges of less than this)
constexpr int PAIR_WARPS = 8;

// Two sets of combinations as one.
__device__ __forceinline__ Best merged(const Best &x, const Best &y)
{
    const bool first = x.mm < y.mm || (x.mm == y.mm && (x.pp < y.pp || (x.pp == y.pp && (x.mate < y.mate ||
                                                                              (x.mate == y.mate && x.pm <= y.pm)))));
    Best b = first ? x : y;
    b.n = x.n + y.n < x.n ? 0xffffffffu : x.n + y.n;
    b.nbest = (x.mm <= y.mm ? x.nbest : 0u) + (y.mm <= x.mm ? y.nbest : 0u);
    return b;
}

__device__ __forceinline__ void write_pair(const Best &B, mica_pair *__restrict__ out)
{
    mica_pair o;
    o.n_concordant = B.n;
    o.n_best = B.n ? B.nbest : 0;
    o.pos_plus = B.n ? B.pp : 0;
    o.pos_minus = B.n ? B.pm : 0;
    o.plus_mate = (uint8_t)(B.n ? B.mate : 0);
    o.mm = (uint8_t)(B.n ? B.mm : 0);
    o.pad = 0;
    *out = o;
}

// A hit's two words (a caller's hits need not lie on 8-byte boundaries).
__device__ __forceinline__ uint64_t hit_word(const Hit *p)
{
    const uint32_t *w = (const uint32_t *)p;
    return (uint64_t)__ldg(w) | ((uint64_t)__ldg(w + 1) << 32);
}

// First hit of the list with pos >= p.
__device__ __forceinline__ uint64_t first_at(const Hit *list, uint64_t n, long long p)
{
    uint64_t L = 0, R = n;
    while (L < R) {
        const uint64_t M = (L + R) >> 1;
        if ((long long)__ldg(&list[M].pos) < p) L = M + 1;
        else R = M;
    }
    return L;
}

// + strand hits of mate `amate` (list A) against - strand hits of the other
// mate (list Bl, its read length mb), by one thread: the partners' positions p
// satisfy lmin <= p + mb - a.pos <= lmax.
__device__ __forceinline__ void pair_lists(const Hit *A, uint64_t na, const Hit *Bl, uint64_t nb, uint32_t mb,
                                           uint32_t lmin, uint32_t lmax, uint32_t amate, Best &B)
{
    for (uint64_t i = 0; i < na; i++) {
        const uint64_t a = hit_word(A + i);
        if ((a >> 32) & 0xffu) continue;
        const long long lo = (long long)(uint32_t)a + (long long)lmin - (long long)mb;
        const long long hi = (long long)(uint32_t)a + (long long)lmax - (long long)mb;
        for (uint64_t j = nb <= PAIR_SMALL ? 0 : first_at(Bl, nb, lo); j < nb; j++) {
            const uint64_t b = hit_word(Bl + j);
            const long long p = (long long)(uint32_t)b;
            if (p > hi) break;
            if (p >= lo && ((b >> 32) & 0xffu) == 1u)
                offer(B, (uint32_t)((a >> 40) & 0xffu) + (uint32_t)((b >> 40) & 0xffu), (uint32_t)a, amate, (uint32_t)b);
        }
    }
}

// The same by a warp.
__device__ __forceinline__ void pair_lists_warp(const Hit *A, uint32_t na, const Hit *Bl, uint32_t nb, uint32_t mb,
                                                uint32_t lmin, uint32_t lmax, uint32_t amate, int lane, Best &B)
{
    for (uint32_t i0 = 0; i0 < na; i0 += 32) {
        uint64_t a = 1ull << 32;
        if (i0 + (uint32_t)lane < na) a = hit_word(A + i0 + lane);
        uint32_t from = 0, size = 0;
        if (((a >> 32) & 0xffu) == 0) {
            const long long lo = (long long)(uint32_t)a + (long long)lmin - (long long)mb;
            const long long hi = (long long)(uint32_t)a + (long long)lmax - (long long)mb;
            from = (uint32_t)first_at(Bl, nb, lo);
            size = max((uint32_t)first_at(Bl, nb, hi + 1), from) - from;
        }
        uint32_t incl = size;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(PFULL, incl, o);
            if (lane >= o) incl += y;
        }
        const uint32_t all = __shfl_sync(PFULL, incl, 31);
        for (uint32_t t0 = 0; t0 < all; t0 += 32) {
            // combination t belongs to the first + strand hit whose running count is above it
            const uint32_t t = t0 + (uint32_t)lane;
            int src = 0;
#pragma unroll
            for (int step = 16; step; step >>= 1)
                if (__shfl_sync(PFULL, incl, src + step - 1) <= t) src += step;
            src = min(src, 31);
            const uint64_t av = __shfl_sync(PFULL, a, src);
            const uint32_t at = __shfl_sync(PFULL, from, src) + t - (__shfl_sync(PFULL, incl, src) - __shfl_sync(PFULL, size, src));
            if (t < all) {
                const uint64_t b = hit_word(Bl + at);
                if (((b >> 32) & 0xffu) == 1u)
                    offer(B, (uint32_t)((av >> 40) & 0xffu) + (uint32_t)((b >> 40) & 0xffu), (uint32_t)av, amate, (uint32_t)b);
            }
        }
    }
}

__global__ void __launch_bounds__(PAIR_WARPS * 32) k_pair(const uint64_t *__restrict__ off, const Hit *__restrict__ hits,
                                                          const uint16_t *__restrict__ len, uint64_t n_pairs,
                                                          uint32_t lmin, uint32_t lmax, mica_pair *__restrict__ out)
{
    // a block takes 256 pairs at a time: those with a few hits by their own
    // threads, the others listed and taken by the block's warps in turn
    __shared__ uint16_t list[PAIR_WARPS * 32];
    __shared__ uint32_t n_list, next;
    const int lane = threadIdx.x & 31;
    for (uint64_t base = blockIdx.x * (uint64_t)(PAIR_WARPS * 32); base < n_pairs;
         base += (uint64_t)gridDim.x * (PAIR_WARPS * 32)) {
        if (threadIdx.x == 0) n_list = next = 0;
        __syncthreads();
        const uint64_t p = base + threadIdx.x;
        if (p < n_pairs) {
            const uint64_t b1 = off[2 * p], b2 = off[2 * p + 1], e2 = off[2 * p + 2];
            if (e2 - b1 <= PAIR_SMALL || e2 - b1 >= PAIR_LARGE) {
                Best B;
                pair_lists(hits + b1, b2 - b1, hits + b2, e2 - b2, len[2 * p + 1], lmin, lmax, 0, B);
                pair_lists(hits + b2, e2 - b2, hits + b1, b2 - b1, len[2 * p], lmin, lmax, 1, B);
                write_pair(B, out + p);
            } else {
                list[atomicAdd(&n_list, 1u)] = (uint16_t)threadIdx.x;
            }
        }
        __syncthreads();
        for (;;) {
            uint32_t i = 0;
            if (lane == 0) i = atomicAdd(&next, 1u);
            i = __shfl_sync(PFULL, i, 0);
            if (i >= n_list) break;
            const uint64_t q = base + list[i];
            const uint64_t b1 = off[2 * q], b2 = off[2 * q + 1], e2 = off[2 * q + 2];
            Best B;
            pair_lists_warp(hits + b1, (uint32_t)(b2 - b1), hits + b2, (uint32_t)(e2 - b2), len[2 * q + 1], lmin, lmax, 0, lane, B);
            pair_lists_warp(hits + b2, (uint32_t)(e2 - b2), hits + b1, (uint32_t)(b2 - b1), len[2 * q], lmin, lmax, 1, lane, B);
            for (int o = 16; o; o >>= 1) {
                Best y;
                y.n = __shfl_xor_sync(PFULL, B.n, o);
                y.nbest = __shfl_xor_sync(PFULL, B.nbest, o);
                y.mm = __shfl_xor_sync(PFULL, B.mm, o);
                y.pp = __shfl_xor_sync(PFULL, B.pp, o);
                y.pm = __shfl_xor_sync(PFULL, B.pm, o);
                y.mate = __shfl_xor_sync(PFULL, B.mate, o);
                B = merged(B, y);
            }
            if (lane == 0) write_pair(B, out + q);
        }
        __syncthreads();
    }
}

}  // namespace
}  // namespace mica

using namespace mica;

extern "C" {

int mica_pair_device(const uint64_t *d_offsets, const mica_hit *d_hits, const uint16_t *d_lengths,
                     uint64_t n_pairs, uint32_t insert_min, uint32_t insert_max, mica_pair *d_out,
                     void *cuda_stream)
{
    if (insert_min > insert_max) return MICA_EINVAL;
    if (n_pairs == 0) return 0;
    if (!d_offsets || !d_hits || !d_lengths || !d_out) return MICA_EINVAL;
    unsigned g = (unsigned)std::min<uint64_t>((n_pairs + PAIR_WARPS * 32 - 1) / (PAIR_WARPS * 32), 152ull * 64);
    k_pair<<<g, PAIR_WARPS * 32, 0, (cudaStream_t)cuda_stream>>>(d_offsets, (const Hit *)d_hits, d_lengths, n_pairs,
                                                      insert_min, insert_max, d_out);
    MICA_CUDA_TRY(cudaGetLastError());
    return 0;
}

int mica_pair_batch(int device, const uint64_t *offsets, const mica_hit *hits, const uint16_t *lengths,
                    uint64_t n_pairs, uint32_t insert_min, uint32_t insert_max, mica_pair *out)
{
    if (insert_min > insert_max) return MICA_EINVAL;
    if (n_pairs == 0) return 0;
    if (!offsets || !lengths || !out) return MICA_EINVAL;
    const uint64_t n_reads = 2 * n_pairs, nh = offsets[n_reads];
    if (nh && !hits) return MICA_EINVAL;
    for (uint64_t r = 0; r < n_reads; r++)
        if (offsets[r] > offsets[r + 1]) return MICA_EINVAL;
    DeviceGuard g(device);
    MICA_CUDA_TRY(cudaSetDevice(device));
    DevBuf doff, dhits, dlen, dout;
    int rc = dev_reserve(doff, (n_reads + 1) * 8);
    if (!rc) rc = dev_reserve(dhits, std::max<uint64_t>(nh, 1) * sizeof(mica_hit));
    if (!rc) rc = dev_reserve(dlen, n_reads * 2);
    if (!rc) rc = dev_reserve(dout, n_pairs * sizeof(mica_pair));
    cudaError_t e = cudaSuccess;
    if (!rc) e = cudaMemcpy(doff.p, offsets, (n_reads + 1) * 8, cudaMemcpyHostToDevice);
    if (!rc && e == cudaSuccess && nh) e = cudaMemcpy(dhits.p, hits, nh * sizeof(mica_hit), cudaMemcpyHostToDevice);
    if (!rc && e == cudaSuccess) e = cudaMemcpy(dlen.p, lengths, n_reads * 2, cudaMemcpyHostToDevice);
    if (!rc && e != cudaSuccess) { set_last_cuda_error(e, "pair upload", __FILE__, __LINE__); rc = MICA_ECUDA; }
    if (!rc) rc = mica_pair_device((const uint64_t *)doff.p, (const mica_hit *)dhits.p, (const uint16_t *)dlen.p,
                                   n_pairs, insert_min, insert_max, (mica_pair *)dout.p, nullptr);
    if (!rc) {
        e = cudaMemcpy(out, dout.p, n_pairs * sizeof(mica_pair), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) { set_last_cuda_error(e, "pair download", __FILE__, __LINE__); rc = MICA_ECUDA; }
    }
    dev_release(doff);
    dev_release(dhits);
    dev_release(dlen);
    dev_release(dout);
    return rc;
}

}  // extern "C"

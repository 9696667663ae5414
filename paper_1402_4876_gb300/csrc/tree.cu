// The search trees the sweep leaves: the nodes of every tree in one frontier
// in global memory, one thread a node (bidir.cu has the scheme search itself,
// and the warp pool that works from it when a small node budget is set).
//
// A tree comes from a seed in a long repeat: an interval of hundreds to tens of
// thousands of rows whose extension is a chain of 100-250 dependent steps with
// small branches.  A lane extends its node, the largest child goes on in the
// lane, and the others wait in the warp's stage in shared memory for idle lanes;
// an interval of a few dozen rows goes on the list of rows to check.  A stage
// that fills, and every node once the launch's nodes are all taken and
// TREE_TAIL more steps are done, goes to the frontier of the next launch, which
// spreads them over all warps again.
//
// A launch stops early when the list of rows to check is nearly full, or the
// next frontier with the nodes not yet taken: the warp that finds it so says
// so, every warp puts its nodes in the frontier, and the warp pool, which checks
// rows itself and has overflow stacks, goes on from all that is left.  Such
// batches have tens of millions of row items (short reads with a large budget,
// reads of a family of a thousand copies).  Going on here instead, with small
// intervals as nodes and the reads of nodes without room given up to the
// one-directional search, took 25.8 ms for 200k reads of 36-60 bp, k = 3, on a
// 64 Mbp genome (now 4.8; the pool alone 3.9) and 21.2 ms for 100k reads of 100
// bp in a family of 1,000 copies at 0.5% (now 9.7).
//
// What bounds it: the longest tree of a block.  Of 17.3 cycles between a warp's
// issues 10.5 are at the barrier before the block's end, 1.7 on global loads (300k x
// 150 bp reads, 64 Mbp genome with repeats).  A step reads two occurrence blocks
// (both loaded whole at once; L2 for a genome of up to some 150 Mbp) and does
// integer work on them.  The warp pool spent 3,000-14,000 cycles a round on its
// stacks and slots, with 1-5 of 32 lanes at work on these trees.  Search kernels
// with the pool in this one's place when it came / now: 100k reads of 100-250 bp
// on a 32 Mbp human-like genome 2.36 / 0.49 ms, 1M mates on a 512 Mbp one 5.8 /
// 3.0 ms, 100k x 250 bp, k = 3 on 16 Mbp 0.53 / 0.54 ms, uneven 1M reads on 64 Mbp
// 1.56 / 1.38 ms.  TREE_TAIL 24 / 48 / 96 / 200 now: 0.82 / 0.70 / 0.61 / 0.49 ms for
// the first of these, 1.88 / 1.65 / 1.51 / 1.38 for the last.
#include <algorithm>

#include "sweep_common.cuh"

namespace mica {
namespace {

constexpr unsigned TFULL = 0xffffffffu;
constexpr int TREE_THREADS = 256;
constexpr int TREE_CTAS = 3;            // per SM
static_assert(TREE_WARPS == 152u * TREE_CTAS * (TREE_THREADS / 32), "warps of a launch");
constexpr uint32_t TREE_TAIL = 200;      // steps of a warp after the launch's nodes are all taken
constexpr uint32_t TREE_REFILL = 8;     // idle lanes of a warp before it takes new nodes
constexpr uint32_t STAGE_LOW = 32;      // staged nodes (items) kept; a step adds at most 96 (128)
constexpr uint32_t STAGE_NODES = 128;
constexpr uint32_t STAGE_ITEMS = 160;

static_assert(STAGE_ITEMS <= 160 && STAGE_NODES + 32 <= 160, "TREE_LAST");

struct TreeStage {
    uint4 node[STAGE_NODES];
    uint4 item[STAGE_ITEMS];
    uint32_t meta[STAGE_NODES];
};

struct TreeArgs {
    OccSide fwd, rev;
    ReadsView rd;
    SearchCtl *ctl;
    Interval *iv;
    uint32_t *iv_cnt;
    uint32_t in_cap;             // nodes `in` may hold (the sweep's counter runs past its own)
    const uint4 *in;             // (task, l, lr, rows)
    const uint32_t *in_meta;
    uint4 *out;
    uint32_t *out_meta;
    uint32_t cap;                // nodes the launch stops at; `out` has room for TREE_LAST more
    uint4 *items;                // rows to check (sweep_common.cuh)
    uint32_t item_cap;           // items the launch stops at
    uint32_t round;
    uint32_t *redo;
    uint32_t verify_min;
    uint32_t tail;               // TREE_TAIL, or a debug limit
};

__device__ __forceinline__ uint32_t tree_C(const OccSide &s, uint32_t c)
{
    return c == 0 ? s.C[0] : c == 1 ? s.C[1] : c == 2 ? s.C[2] : s.C[3];
}

// A node for the next launch.  (One past the end, which a launch that stops in
// time has none of, gives its read up to the persistent kernel.)
__device__ __forceinline__ void push_node(const TreeArgs &a, uint32_t q, uint32_t task, uint32_t l, uint32_t lr,
                                          uint32_t sz, uint32_t meta)
{
    if (q < a.cap + TREE_LAST) {
        a.out[q] = make_uint4(task, l, lr, sz);
        a.out_meta[q] = meta;
    } else {
        const uint32_t rid = task >> 1, bit = 1u << (rid & 31);
        if (!(atomicOr(&a.redo[rid >> 5], bit) & bit)) atomicAdd(&a.ctl->redo_reads, 1u);
    }
}

// The staged items to their list; false when it is nearly full.
__device__ __forceinline__ bool flush_items(const TreeArgs &a, const TreeStage &S, uint32_t n, int lane)
{
    uint32_t at = 0;
    if (lane == 0) at = atomicAdd(&a.ctl->row_items, n);
    at = __shfl_sync(TFULL, at, 0);
    for (uint32_t i = lane; i < n; i += 32) a.items[at + i] = S.item[i];
    __syncwarp();
    return at + n < a.item_cap;
}

// The staged nodes [from, n) to the frontier; false when it is nearly full with
// the launch's nodes that are not yet taken.
__device__ __forceinline__ bool flush_nodes(const TreeArgs &a, const TreeStage &S, uint32_t from, uint32_t n,
                                            uint32_t ntasks, int lane)
{
    uint32_t at = 0, left = 0;
    if (lane == 0) {
        const unsigned long long head = *(volatile unsigned long long *)&a.ctl->task_head;
        at = atomicAdd(&a.ctl->fr_count, n - from);
        left = head < ntasks ? ntasks - (uint32_t)head : 0u;
    }
    at = __shfl_sync(TFULL, at, 0);
    left = __shfl_sync(TFULL, left, 0);
    for (uint32_t i = from + lane; i < n; i += 32) {
        const uint4 x = S.node[i];
        push_node(a, at + i - from, x.x, x.y, x.z, x.w, S.meta[i]);
    }
    __syncwarp();
    return at + (n - from) + left < a.cap;
}

__global__ void __launch_bounds__(TREE_THREADS, TREE_CTAS) k_tree(const TreeArgs a)
{
    extern __shared__ uint4 tree_smem[];
    SearchCtl *ctl = a.ctl;
    const uint32_t ntasks = (uint32_t)min(*(volatile unsigned long long *)&ctl->ntasks, (unsigned long long)a.in_cap);
    const unsigned stopped = *(volatile unsigned *)&ctl->stop;
    if (ntasks == 0 || *(volatile unsigned *)&ctl->error || (stopped && stopped != a.round)) return;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    TreeStage &S = reinterpret_cast<TreeStage *>(tree_smem)[threadIdx.x >> 5];
    // nodes a warp takes at a time: no more than its part of the launch's
    const uint32_t share = max(1u, min(32u, ntasks / (gridDim.x * (TREE_THREADS / 32))));
    // with at least half as many nodes as the launch has lanes (TREE_SPLIT_FEW's comment)
    const uint32_t few = 2ull * ntasks >= (unsigned long long)gridDim.x * TREE_THREADS ? TREE_SPLIT_FEW : TREE_SPLIT_LEFT;
    bool active = false, more = true;
    uint32_t task = 0, l = 0, lr = 0, sz = 0, lim = 0, A = 0, B = 0, d = 0, d0 = 0, j = 0, m = 0, k = 0;
    unsigned long long bounds = 0;
    const uint32_t *w = nullptr;
    uint32_t c_nodes = 0, c_blocks = 0, nn = 0, ni = 0, tail = 0;   // staged nodes, staged items
    // the launch stops: no more nodes are taken, and the next step hands on what the warp has
    const auto halt = [&]() {
        more = false;
        tail = 0x7fffffffu;
        if (lane == 0) *(volatile unsigned *)&ctl->stop = a.round;
    };
    if (__shfl_sync(TFULL, lane == 0 ? *(volatile unsigned *)&ctl->row_items : 0u, 0) >= a.item_cap) halt();
    for (;;) {
        // idle lanes take staged nodes, then the launch's
        unsigned idle = __ballot_sync(TFULL, !active);
        bool fresh = false;
        uint4 it = make_uint4(0, 0, 0, 0);
        uint32_t meta = 0;
        if (idle && nn) {
            const uint32_t n = min(nn, (uint32_t)__popc(idle)), r = __popc(idle & lt);
            if (!active && r < n) {
                it = S.node[nn - 1 - r];
                meta = S.meta[nn - 1 - r];
                fresh = true;
            }
            nn -= n;
            idle = __ballot_sync(TFULL, !active && !fresh);
            __syncwarp();
        }
        if (more && (idle == TFULL || __popc(idle) >= TREE_REFILL)) {
            const uint32_t n = min((uint32_t)__popc(idle), share);
            unsigned long long t0 = 0;
            unsigned stop = 0;
            if (lane == 0) {
                stop = *(volatile unsigned *)&ctl->stop;
                t0 = atomicAdd(&ctl->task_head, (unsigned long long)n);
            }
            t0 = __shfl_sync(TFULL, t0, 0);
            more = t0 + n < ntasks;
            if (__shfl_sync(TFULL, stop, 0)) halt();
            const uint32_t r = __popc(idle & lt);
            if (!active && !fresh && r < n && t0 + r < ntasks) {
                it = a.in[t0 + r];
                meta = a.in_meta[t0 + r];
                fresh = true;
            }
        }
        if (fresh) {
            task = it.x; l = it.y; lr = it.z; sz = it.w;
            lim = max(few, sz - (sz + 7u) / 8u);
            A = bm_a(meta); B = bm_b(meta); d = bm_d(meta); d0 = bm_d0(meta); j = bm_j(meta);
            const uint32_t rid = task >> 1;
            m = a.rd.len[rid];
            k = a.rd.k[rid];
            w = a.rd.words + a.rd.word_off[rid];
            bounds = pack_bounds(m, m >= k + 1 ? k + 1 : 1u);
            // the node of a read already given up is not continued
            active = !((a.redo[rid >> 5] >> (rid & 31)) & 1u);
        }
        if (!__any_sync(TFULL, active)) {
            if (!more && nn == 0) break;
            continue;
        }
        if (!more && ++tail > a.tail) {
            // the rest to the next launch (or to the warp pool)
            const unsigned act = __ballot_sync(TFULL, active);
            if (active) {
                const uint32_t q = nn + __popc(act & lt);
                S.node[q] = make_uint4(task, l, lr, sz);
                S.meta[q] = bd_meta(0, A, B, d, d0, j);
            }
            nn += __popc(act);
            __syncwarp();
            if (!flush_nodes(a, S, 0, nn, ntasks, lane)) halt();
            break;
        }
        uint32_t cl[4] = {0, 0, 0, 0}, clr[4] = {0, 0, 0, 0}, cs[4] = {0, 0, 0, 0};
        uint32_t leafmask = 0, nodemask = 0, itemmask = 0, d0mis = 0, d0hit = 0, nA = 0, nB = 0, base = 0, pick = 0;
        if (active) {
            const bool left = A > 0;
            const uint32_t pos = left ? A - 1 : B, q = (task & 1u) ? m - 1 - pos : pos;
            const uint32_t word = __ldg(w + (q >> 4));
            const OccSide &sd = left ? a.fwd : a.rev;
            const uint32_t pl = left ? l : lr;              // interval on the side being extended
            uint32_t ol[4], orr[4];
            c_blocks += occ_pair(sd, pl, pl + sz, ol, orr);
            c_nodes++;
            base = (word >> (2u * (q & 15u))) & 3u;
            if (task & 1u) base = 3u - base;
            nA = left ? pos : 0;
            nB = left ? B : pos + 1;
            const bool hit = bd_allowed(j, A, pos, bounds, k, d, d0, 0, d0hit);
            const bool mis = bd_allowed(j, A, pos, bounds, k, d, d0, 1, d0mis);
            // the other side's interval start: rows of lower symbols (and a $) come first
            uint32_t acc = (left ? lr : l) + ((sd.dollar_row >= pl && sd.dollar_row < pl + sz) ? 1u : 0u);
            const bool whole = nA == 0 && nB == m;
            const bool checkable = a.verify_min && nB - nA >= a.verify_min && m - (nB - nA) >= BD_VERIFY_LEFT;
            const uint32_t split = nA ? min(TREE_SPLIT_LEFT, lim) : TREE_SPLIT_RIGHT;
            uint32_t most = 0;
#pragma unroll
            for (uint32_t c = 0; c < 4; c++) {
                const uint32_t n_c = orr[c] - ol[c];
                if (n_c > 0 && (c == base ? hit : mis)) {
                    const uint32_t start = tree_C(sd, c) + ol[c];
                    cl[c] = left ? start : acc;
                    clr[c] = left ? acc : start;
                    cs[c] = n_c;
                    if (whole) leafmask |= 1u << c;
                    else if (checkable && n_c <= split) itemmask |= 1u << c;
                    else { nodemask |= 1u << c; most = max(most, n_c); }
                }
                acc += n_c;
            }
            active = nodemask != 0;
            if (active) {
                // the largest child goes on here
#pragma unroll
                for (uint32_t c = 0; c < 4; c++)
                    if ((nodemask >> c & 1u) && cs[c] == most) pick = c;
                nodemask &= ~(1u << pick);
                l = pick == 0 ? cl[0] : pick == 1 ? cl[1] : pick == 2 ? cl[2] : cl[3];
                lr = pick == 0 ? clr[0] : pick == 1 ? clr[1] : pick == 2 ? clr[2] : clr[3];
                sz = most;
            }
        }
        // leaves to the interval buffer; nodes and row items to the stage
        const uint32_t packed = __popc(leafmask) | (__popc(nodemask) << 8) | (__popc(itemmask) << 16);
        if (__any_sync(TFULL, packed)) {
            uint32_t incl = packed;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(TFULL, incl, o);
                if (lane >= o) incl += y;
            }
            const uint32_t all = __shfl_sync(TFULL, incl, 31), excl = incl - packed;
            uint32_t at_leaf = 0;
            if (all & 0xffu) {
                if (lane == 0) at_leaf = atomicAdd(&ctl->iv_count, all & 0xffu);
                at_leaf = __shfl_sync(TFULL, at_leaf, 0) + (excl & 0xffu);
            }
            uint32_t at_node = nn + ((excl >> 8) & 0xffu), at_item = ni + (excl >> 16);
            if (packed) {
                const uint32_t rid = task >> 1;
                if (leafmask) atomicAdd(&a.iv_cnt[rid], __popc(leafmask));
                uint32_t ctx = 0, ex = 0;
                if (itemmask) {
                    const uint32_t aj = bound_at(bounds, j);   // (only a piece's scheme is checkable)
                    ex = nA > aj ? min(16u, nA - aj) : 0u;
                    ctx = read_context(w, task & 1u, m, nA);
                }
#pragma unroll
                for (uint32_t c = 0; c < 4; c++) {
                    const uint32_t dn = c == base ? d : d + 1;
                    if (leafmask >> c & 1u) {
                        if (at_leaf < ctl->iv_cap) {
                            Interval x;
                            x.read = rid; x.meta = dn | ((task & 1u) << 2); x.l = cl[c]; x.r = cl[c] + cs[c];
                            a.iv[at_leaf] = x;
                        } else {
                            atomicOr(&ctl->error, ERR_IV_OVERFLOW);
                        }
                        at_leaf++;
                    }
                    if (itemmask >> c & 1u)
                        S.item[at_item++] = make_uint4(cl[c], task, item_meta(cs[c], j, ex, k, nA, k - dn), ctx);
                    if (nodemask >> c & 1u) {
                        S.node[at_node] = make_uint4(task, cl[c], clr[c], cs[c]);
                        S.meta[at_node++] = bd_meta(0, nA, nB, dn, c == base ? d0hit : d0mis, j);
                    }
                }
            }
            nn += (all >> 8) & 0xffu;
            ni += all >> 16;
            __syncwarp();
            if (nn > STAGE_LOW) {
                if (!flush_nodes(a, S, STAGE_LOW, nn, ntasks, lane)) halt();
                nn = STAGE_LOW;
            }
            if (ni > STAGE_LOW) {
                if (!flush_items(a, S, ni, lane)) halt();
                ni = 0;
            }
        }
        if (active) {   // the continuing child
            A = nA;
            B = nB;
            d0 = pick == base ? d0hit : d0mis;
            d += pick == base ? 0u : 1u;
        }
    }
    if (ni && !flush_items(a, S, ni, lane)) halt();
    c_nodes = __reduce_add_sync(TFULL, c_nodes);
    c_blocks = __reduce_add_sync(TFULL, c_blocks);
    if (lane == 0 && c_nodes) {
        atomicAdd(&ctl->nodes, (unsigned long long)c_nodes);
        atomicAdd(&ctl->rank_blocks, (unsigned long long)c_blocks);
        atomicAdd(&ctl->lane_ops, (unsigned long long)c_nodes);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&ctl->done_ctas, 1u) == gridDim.x - 1) {
        const unsigned long long head = *(volatile unsigned long long *)&ctl->task_head;
        const bool stop = *(volatile unsigned *)&ctl->stop != 0;
        ctl->left_from = (uint32_t)min(head, (unsigned long long)ntasks);
        ctl->left_to = ntasks;
        end_round(ctl, a.cap + TREE_LAST);
        if (stop) ctl->unfinished |= 8u;
    }
}

}  // namespace

// One launch of the trees, the round-th: the nodes of `in` (their number in
// ctl->ntasks, at most in_cap of them written), their children to `out`, which has room for cap + TREE_LAST;
// items has room for item_cap.  tail: steps after the launch's nodes are all
// taken (0: TREE_TAIL).
int launch_tree(const OccSide &fwd, const OccSide &rev, Workspace &w, const ReadsView &rd, uint32_t round,
                const uint4 *in, const uint32_t *in_meta, uint32_t in_cap, uint4 *out, uint32_t *out_meta, uint32_t cap,
                uint4 *items, uint32_t item_cap, uint32_t *redo, uint32_t verify_min, uint32_t tail, cudaStream_t s)
{
    TreeArgs a;
    a.fwd = fwd;
    a.rev = rev;
    a.rd = rd;
    a.ctl = (SearchCtl *)w.ctl.p;
    a.iv = (Interval *)w.iv.p;
    a.iv_cnt = (uint32_t *)w.iv_cnt.p;
    a.in = in;
    a.in_meta = in_meta;
    a.in_cap = in_cap;
    a.out = out;
    a.out_meta = out_meta;
    a.cap = cap;
    a.items = items;
    a.item_cap = !verify_min ? 0xffffffffu : item_cap > TREE_LAST ? item_cap - TREE_LAST : 0u;
    a.round = round;
    a.redo = redo;
    a.verify_min = verify_min;
    a.tail = tail ? tail : TREE_TAIL;
    constexpr size_t smem = sizeof(TreeStage) * (TREE_THREADS / 32);
    MICA_CUDA_TRY(cudaFuncSetAttribute(k_tree, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_tree<<<152 * TREE_CTAS, TREE_THREADS, smem, s>>>(a);
    MICA_CUDA_TRY(cudaGetLastError());
    return 0;
}

}  // namespace mica

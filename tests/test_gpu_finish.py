"""The kernels that finish reads of different sizes (a thread, a warp, a block,
a block for long interval lists, the host's loop) and pair mates with few or
many hits, at the sizes where one hands over to the next."""
import numpy as np
import pytest

import oracle
import synth
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


def _genome_with_copies(copies, unit=60, gap=41, seed=3):
    """`copies` copies of one random unit, `gap` random bases apart, in a random genome."""
    rng = np.random.default_rng(seed)
    u = rng.integers(0, 4, size=unit, dtype=np.uint8)
    parts = [rng.integers(0, 4, size=500, dtype=np.uint8)]
    for _ in range(copies):
        parts += [u, rng.integers(0, 4, size=gap, dtype=np.uint8)]
    return np.concatenate(parts), u


@pytest.mark.parametrize("copies", [1, 2, 8, 9, 31, 33, 255, 256, 257, 4095, 4097])
@pytest.mark.parametrize("full_sa", [True, False])
def test_hit_counts_around_the_kernels_limits(copies, full_sa):
    """A read with exactly `copies` exact placements (spread wider than the
    counting sort's span from about 40 and 200 copies up), beside an ordinary one, under caps below, at
    and above that number."""
    g, u = _genome_with_copies(copies)
    reads = [u, (3 - u)[::-1].copy(), g[:60].copy()]
    b = gc.batch_from_reads(reads, [0, 0, 1])
    fm = oracle.FMIndex(g)
    idx = gc.mica().Index.build(synth.to_acgt_bytes(g), kmer_q=10, sa_sample=8, full_sa=full_sa)
    for cap in sorted({1, max(1, copies - 1), copies, copies + 1, 0}):
        gc.assert_same(idx.align_batch(b, hit_cap=cap), fm.align(b, cap=cap), f"copies {copies} cap {cap}")
    idx.free()


@pytest.mark.parametrize("cap", [1, 10, 255, 1000, 4096, 5000, 70_000, 0])
def test_long_interval_lists_under_caps(cap):
    """Reads inside a diverged array have thousands of one-row intervals in
    several (d, strand) classes, more than a warp or a small block holds."""
    rng = np.random.default_rng(11)
    core = np.resize(np.array([0, 1, 2], np.uint8), 30_000)
    mut = rng.random(core.size) < 0.03
    core[mut] = (core[mut] + rng.integers(1, 4, size=int(mut.sum()))) & 3
    g = np.concatenate([rng.integers(0, 4, 3_000).astype(np.uint8), core])
    reads = [g[3_000 + 700 * i: 3_000 + 700 * i + 36].copy() for i in range(12)]
    b = gc.batch_from_reads(reads, [0, 1, 2, 3] * 3)
    idx = gc.mica().Index.build(synth.to_acgt_bytes(g), kmer_q=10, sa_sample=8)
    gc.assert_same(idx.align_batch(b, hit_cap=cap), oracle.FMIndex(g).align(b, cap=cap), f"cap {cap}")
    idx.free()


@pytest.mark.parametrize("n", [1, 511, 512, 513, 1025])
def test_batch_sizes_around_a_tile(n):
    """Batches that end before, at and after a tile of the prefix sums."""
    g = synth.uniform_genome(50_000, 5)
    rng = np.random.default_rng(n)
    b = synth.sample_reads(g, rng.integers(20, 90, n), rng.integers(0, 3, n), rng, subs="rate", sub_rate=0.02)
    idx = gc.mica().Index.build(synth.to_acgt_bytes(g.codes), kmer_q=9, sa_sample=8)
    gc.assert_same(idx.align_batch(b, hit_cap=3), oracle.FMIndex(g.codes).align(b, cap=3), f"n {n}")
    idx.free()


@pytest.mark.parametrize("sizes", [(4, 4), (4, 5), (1, 40), (33, 64), (300, 500), (0, 9), (1000, 1000)])
def test_pairs_of_many_hits(sizes):
    """Mates with few and many hits (some windows hold every hit of the other
    mate), ties included."""
    rng = np.random.default_rng(sum(sizes))
    m = gc.mica()
    for span, lo, hi in ((400, 0, 5_000), (4_000, 300, 700), (3_000, 450, 450)):
        lists = []
        for _ in range(3):
            for n in sizes:
                pick = rng.choice(2 * span, size=min(n, 2 * span), replace=False)
                lists.append(sorted((int(x) // 2, int(x) % 2, int(rng.integers(0, 3))) for x in pick))
        off = np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(np.uint64)
        hits = np.zeros(int(off[-1]), dtype=m.HIT_DTYPE)
        for j, h in enumerate(h for x in lists for h in x):
            hits[j] = (*h, 0)

        class R:
            offsets = off

            @staticmethod
            def as_tuples(i):
                return lists[i]

            @staticmethod
            def hits_of(i):
                return lists[i]
        R.hits = hits
        lens = np.array([100, 150] * 3, np.uint16)
        got = [(int(x["n_concordant"]), int(x["n_best"]), int(x["pos_plus"]), int(x["pos_minus"]),
                int(x["plus_mate"]), int(x["mm"])) for x in m.pair_batch(R, lens, lo, hi)]
        assert got == oracle.pair(R, lens, lo, hi), (sizes, span)


def test_invalid_device_batches_are_refused_in_the_captured_batch():
    """The check of a device batch runs inside the captured batch: a read of no
    bases, a budget of 4 and an offset past the words are refused every time,
    and the valid batch in the same buffers is not."""
    import torch
    m = gc.mica()
    g = synth.uniform_genome(20_000, 8)
    rng = np.random.default_rng(2)
    b = synth.sample_reads(g, np.full(300, 50), np.full(300, 1), rng, subs="rate", sub_rate=0.01)
    idx = m.Index.build(synth.to_acgt_bytes(g.codes), kmer_q=8, sa_sample=8)
    d = [torch.from_numpy(b.words.view(np.int32)).cuda(), torch.from_numpy(b.word_off.view(np.int64)).cuda(),
         torch.from_numpy(b.lengths.view(np.int16)).cuda(), torch.from_numpy(b.k).cuda()]
    want = oracle.FMIndex(g.codes).align(b, cap=1000)
    for which, value in ((2, 0), (3, 4), (1, 1 << 40), (2, 300)):
        for _ in range(2):
            keep = d[which][7].clone()
            d[which][7] = value
            with pytest.raises(m.MicaError) as e:
                idx.align_device(*d, b.n)
            assert e.value.code == m.MICA_EINVAL
            d[which][7] = keep
            t, o, h = idx.align_device(*d, b.n).tensors()
            got = m.Result(t.cpu().numpy().view(np.uint64), o.cpu().numpy().view(np.uint64),
                           h.cpu().numpy().view(m.HIT_DTYPE))
            gc.assert_same(got, want, f"{which} {value}")
    idx.free()


@pytest.mark.parametrize("full_sa", [True, False])
def test_more_trees_than_the_frontier_holds(full_sa):
    """300,000 reads whose seeds are too short to be checked (40 bases in four
    pieces) leave more first nodes than the frontier's 2^20: the rest go to the
    warp pool as tasks.  Every result equals the persistent kernel's, on repeated
    calls, and a sample the oracle's."""
    g = synth.uniform_genome(300_000, 21)
    rng = np.random.default_rng(4)
    b = synth.sample_reads(g, np.full(300_000, 40), np.full(300_000, 3), rng, subs="rate", sub_rate=0.02)
    idx = gc.mica().Index.build(synth.to_acgt_bytes(g.codes), kmer_q=10, sa_sample=8, full_sa=full_sa)
    want = idx.align_batch(b, hit_cap=10, kernel="persistent")
    for call in range(2):
        gc.assert_same(idx.align_batch(b, hit_cap=10), want, f"call {call}")
    assert idx.stats()["fallback_reads"] == 0
    some = b.subset(np.arange(0, b.n, 600))
    gc.assert_same(idx.align_batch(some, hit_cap=10), oracle.FMIndex(g.codes).align(some, cap=10), "sample")
    idx.free()


@pytest.mark.parametrize("m,k", [(1, 0), (2, 3), (3, 3), (4, 3), (11, 0), (12, 0), (20, 1), (32, 1), (33, 1), (48, 3), (256, 3)])
@pytest.mark.parametrize("full_sa", [True, False])
def test_tree_shapes(m, k, full_sa):
    """Reads shorter than k + 1 bases (one tree from the full interval), whole-read
    seeds, pieces around the verify threshold and the longest reads, inside an
    exact tandem array, at both ends of the genome and elsewhere."""
    rng = np.random.default_rng(100 * m + k)
    g = np.concatenate([rng.integers(0, 4, 3_000).astype(np.uint8), np.resize(rng.integers(0, 4, 7).astype(np.uint8), 4_000),
                        rng.integers(0, 4, 3_000).astype(np.uint8)])
    at = [0, g.size - m, 1_500, 3_500, 4_200, 6_990, 8_000]
    reads = []
    for i, a in enumerate(at):
        r = g[a:a + m].copy()
        if m > 20:
            synth.substitute(r, rng.choice(m, size=i % (k + 1), replace=False), rng)
        reads.append(r if i % 2 else (3 - r)[::-1].copy())
    b = gc.batch_from_reads(reads, [k] * len(reads))
    idx = gc.mica().Index.build(synth.to_acgt_bytes(g), kmer_q=8, sa_sample=8, full_sa=full_sa)
    for cap in (0, 50):
        gc.assert_same(idx.align_batch(b, hit_cap=cap), oracle.FMIndex(g).align(b, cap=cap), f"m {m} k {k} cap {cap}")
    idx.free()

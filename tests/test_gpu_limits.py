"""The bidirectional search's default path (seed sweep, trees from a frontier, row
checks) with each of its lists and launch limits made to run out: results stay
the oracle's, alone and in combination, on repeated calls."""
import functools

import numpy as np
import pytest

import oracle
import synth
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu

# Of the row items' list the trees leave this many for what they staged before it was full.
LAST_FLUSHES = 152 * 3 * 8 * 160


def _copies(unit, n, div, rng):
    """n copies of a unit at divergence div, 20-60 random bases apart."""
    parts = []
    for _ in range(n):
        u = unit.copy()
        hit = rng.random(u.size) < div
        u[hit] = (u[hit] + rng.integers(1, 4, int(hit.sum()))) & 3
        parts += [u, rng.integers(0, 4, int(rng.integers(20, 60)))]
    return np.concatenate(parts)


@functools.lru_cache(maxsize=None)
def _inputs():
    """A genome of repeats whose seeds name a few dozen rows (row items), hundreds
    (trees) and thousands (trees of many branches), reads of each and two batches
    of them in different orders."""
    rng = np.random.default_rng(31)
    unit = lambda n: rng.integers(0, 4, n)
    parts = [unit(30_000), _copies(unit(300), 40, 0.0, rng), _copies(unit(250), 300, 0.03, rng),
             _copies(np.resize(unit(7), 5_000), 1, 0.03, rng), unit(5_000)]
    g = np.concatenate(parts).astype(np.uint8)
    at = np.cumsum([0] + [p.size for p in parts])
    reads, ks = [], []

    def some(i, count, m, k):
        for _ in range(count):
            a = int(rng.integers(at[i], min(at[i + 1], g.size - m)))
            r = g[a:a + m].copy()
            hit = rng.random(m) < 0.01
            r[hit] = (r[hit] + rng.integers(1, 4, int(hit.sum()))) & 3
            reads.append(r if rng.random() < 0.5 else (3 - r)[::-1].copy())
            ks.append(k)

    for k in (0, 1, 2, 3):
        some(0, 20, 100, k)
        some(1, 120, 101, k)
        some(2, 100, 150, k)
        some(3, 12, 60, k)
    some(2, 60, 33, 3)      # pieces too short for a row check: every seed is a tree
    some(0, 20, 3, 3)       # no pieces: one tree from the full interval
    order = rng.permutation(len(reads))
    a = gc.batch_from_reads([reads[i] for i in order], [ks[i] for i in order])
    order = order[::-1]
    b = gc.batch_from_reads([reads[i] for i in order], [ks[i] for i in order])
    fm = oracle.FMIndex(g)
    return g, a, b, {cap: fm.align(a, cap=cap) for cap in (0, 20)}


def _index(full_sa=True):
    return gc.mica().Index.build(synth.to_acgt_bytes(_inputs()[0]), kmer_q=12, sa_sample=8, full_sa=full_sa)


def _path_is_the_trees(idx):
    assert idx.stats()["warp_rounds"] == 0, "the warp pool took part"


@pytest.mark.parametrize("row_items", [1, 33, 500, LAST_FLUSHES + 1, LAST_FLUSHES + 2_000])
def test_the_row_item_list_runs_out(row_items):
    """A list with room for fewer row items than the sweep (up to 500) or the
    trees want, after a batch of the same reads in another order has filled
    it: what finds no room is searched otherwise, and no entry that another
    batch left behind is looked at."""
    g, a, b, want = _inputs()
    idx = _index()
    idx.align_batch(b, hit_cap=20)
    gc.assert_same(idx.align_batch(a, hit_cap=20), want[20], "built-in limits")
    _path_is_the_trees(idx)
    free = idx.stats()
    assert free["verified"] > 0
    idx.align_batch(b, hit_cap=20)
    idx.debug_search_limits(row_items=row_items)
    for call in range(2):
        for cap in (20, 0):
            gc.assert_same(idx.align_batch(a, hit_cap=cap), want[cap], f"items {row_items} call {call} cap {cap}")
            assert idx.stats()["fallback_reads"] == 0
    assert idx.stats()["nodes"] > free["nodes"]       # what found no room was extended instead
    idx.free()


@pytest.mark.parametrize("full_sa", [True, False])
@pytest.mark.parametrize("limits", [
    dict(nodes=64), dict(steps=1), dict(rounds=1, steps=1), dict(rounds=2, steps=2), dict(nodes=4096, steps=3),
    dict(nodes=400, rounds=1, steps=1),      # tasks left to the warp pool, and trees that outlast their rounds
    dict(nodes=64, rounds=1, steps=1), dict(nodes=400, rounds=3, steps=2, row_items=40),
    dict(nodes=4, rounds=64, steps=1, row_items=1)], ids=str)
def test_limits_of_the_trees(limits, full_sa):
    """The frontier's nodes (first nodes past its end are the warp pool's tasks,
    and a launch whose children fill it stops), a launch's steps, the launches, and these
    together: every read's hits are the oracle's, through a call that captures,
    one that replays, and the pipelined calls."""
    _, a, b, want = _inputs()
    idx = _index(full_sa)
    idx.align_batch(b, hit_cap=20)
    idx.debug_search_limits(**limits)
    for cap in (20, 0):
        for call in range(2):
            gc.assert_same(idx.align_batch(a, hit_cap=cap), want[cap], f"{limits} cap {cap} call {call}")
    gc.assert_same(idx.collect(idx.submit_batch(a, hit_cap=20)), want[20], f"{limits} pipelined")
    if "rounds" in limits and "nodes" not in limits:
        assert idx.stats()["fallback_reads"] > 0
    idx.debug_search_limits()
    gc.assert_same(idx.align_batch(a, hit_cap=20), want[20], "built-in limits again")
    idx.free()


@pytest.mark.parametrize("budget", [8, 200, 512, 1023])
def test_runs_return_to_a_full_stack(budget):
    """The warp pool: short reads with a large budget fill a warp's stack with
    children of several rows while other lanes' runs (nodes whose rows all
    continue alike) end early and go back to it.  Which lanes meet depends on
    the launch, so two batches are searched 80 times each; the result is the
    persistent kernel's each time."""
    g = synth.genome_64m(1 << 24)
    rng = np.random.default_rng(78)
    batches = [synth.sample_reads(g, rng.integers(36, 61, 50_000), np.full(50_000, 3), rng, subs="rate", sub_rate=0.01,
                                  repeat_frac=0.3) for _ in range(2)]
    idx = gc.mica().Index.build(synth.to_acgt_bytes(g.codes), kmer_q=12, sa_sample=16)
    for b in batches:
        idx.set_tuning()
        want = idx.align_batch(b, hit_cap=10, kernel="persistent")
        idx.set_tuning(bidir_budget=budget)
        for call in range(80):
            gc.assert_same(idx.align_batch(b, hit_cap=10), want, f"budget {budget} call {call}")
            assert idx.stats()["warp_rounds"] > 0
    idx.free()


def _family(copies, div):
    """A 4 Mbp genome with a family of 3 kbp copies at divergence div, and reads inside them."""
    rng = np.random.default_rng(copies)
    g = rng.integers(0, 4, 1 << 22).astype(np.uint8)
    unit, at = rng.integers(0, 4, 3_000), rng.permutation((1 << 22) // 3_500 - 1)[:copies] * 3_500
    for s in at:
        u = unit.copy()
        hit = rng.random(u.size) < div
        u[hit] = (u[hit] + rng.integers(1, 4, int(hit.sum()))) & 3
        g[s:s + 3_000] = u
    return synth.Genome(g, [(int(s), int(s) + 3_000, "") for s in at])


@pytest.mark.parametrize("case", ["short_k3", "short_k2", "family_1000", "lean_short"])
def test_more_work_than_the_lists_hold(case):
    """Batches whose trees want several times the row items, or nodes, that the
    lists hold: the launch stops in time and the warp pool takes what is left,
    so no read is given up; results are the persistent kernel's."""
    rng = np.random.default_rng(5)
    if case == "family_1000":
        g, n, lo, hi, k, inside = _family(1_000, 0.005), 30_000, 100, 100, 2, 1.0
    else:
        g = synth.genome_64m(1 << 24)
        n, lo, hi, k, inside = {"short_k3": (50_000, 36, 36, 3, 0.2), "short_k2": (200_000, 30, 30, 2, 0.0),
                                "lean_short": (100_000, 24, 24, 2, 0.0)}[case]
    b = synth.sample_reads(g, rng.integers(lo, hi + 1, n), np.full(n, k), rng, subs="rate", sub_rate=0.01, repeat_frac=inside)
    idx = gc.mica().Index.build(synth.to_acgt_bytes(g.codes), full_sa=case != "lean_short")
    want = idx.align_batch(b, hit_cap=10, kernel="persistent")
    for call in range(3):
        gc.assert_same(idx.align_batch(b, hit_cap=10), want, f"{case} call {call}")
        assert idx.stats()["fallback_reads"] == 0
    idx.free()


@pytest.mark.parametrize("rows", [1, 15, 16, 17, 31, 32, 33, 64, 65])
def test_row_items_of_few_and_many_rows(rows):
    """Row items at the size up to which several share a warp's look, at the
    sweep's sizes, and mixed: families of `rows` and of half as many copies,
    whose copies differ in few bases, some at the genome's very ends."""
    rng = np.random.default_rng(rows)
    parts, marks = [], []
    for copies in (rows, max(1, rows // 2), rows):
        unit = rng.integers(0, 4, 220)
        for _ in range(copies):
            u = unit.copy()
            hit = rng.random(u.size) < 0.01
            u[hit] = (u[hit] + rng.integers(1, 4, int(hit.sum()))) & 3
            marks.append(sum(p.size for p in parts))
            parts += [u, rng.integers(0, 4, int(rng.integers(0, 30)))]
    g = np.concatenate(parts).astype(np.uint8)
    reads, ks = [], []
    for i in range(400):
        m = int(rng.integers(24, 180))
        a = min(int(marks[i % len(marks)] + rng.integers(0, 220 - min(m, 219))), g.size - m)
        a = {0: 0, 1: g.size - m}.get(i, a)
        r = g[a:a + m].copy()
        hit = rng.random(m) < 0.01
        r[hit] = (r[hit] + rng.integers(1, 4, int(hit.sum()))) & 3
        reads.append(r if i % 2 else (3 - r)[::-1].copy())
        ks.append(i % 4)
    b = gc.batch_from_reads(reads, ks)
    fm = oracle.FMIndex(g)
    idx = gc.mica().Index.build(synth.to_acgt_bytes(g), kmer_q=12, sa_sample=8)
    for cap in (0, 5):
        gc.assert_same(idx.align_batch(b, hit_cap=cap), fm.align(b, cap=cap), f"rows {rows} cap {cap}")
        _path_is_the_trees(idx)
    assert idx.stats()["verified"] > 0
    idx.free()


@pytest.mark.parametrize("copies", [64, 65, 200, 256, 257])
@pytest.mark.parametrize("n", [300, 30_000])
def test_exact_copies_of_few_and_many_reads(copies, n):
    """Reads inside exact copies: in a batch whose trees fill the GPU's lanes their
    rows stay one interval (not a leaf each), in a small one they are told
    apart; results are the persistent kernel's either way, under a cap and
    without."""
    g = _family(copies, 0.0)
    rng = np.random.default_rng(n)
    b = synth.sample_reads(g, np.full(n, 60), np.full(n, 2), rng, subs="rate", sub_rate=0.01, repeat_frac=1.0)
    idx = gc.mica().Index.build(synth.to_acgt_bytes(g.codes))
    for cap in (10, 0):
        want = idx.align_batch(b, hit_cap=cap, kernel="persistent")
        gc.assert_same(idx.align_batch(b, hit_cap=cap), want, f"cap {cap}")
        _path_is_the_trees(idx)
        if n == 30_000 and copies > 64:
            assert idx.stats()["intervals"] < 8 * n
    idx.free()


@pytest.mark.parametrize("cap", [1, 9, 10, 31, 255, 256])
def test_reads_over_their_cap_with_one_interval_or_a_few(cap):
    """Reads over their cap whose lists hold one interval, as many as a warp's
    lanes, and one more than that."""
    rng = np.random.default_rng(cap)
    parts, reads = [rng.integers(0, 4, 800)], []
    for copies, variants in ((300, 1), (9, 31), (9, 32), (9, 33), (40, 64), (2, 65), (5, 3)):
        unit = rng.integers(0, 4, 80)
        reads.append(unit)
        for v in range(variants):             # each its own interval: a base of its own, or none
            u = unit.copy()
            if v:
                u[v % 80] = (u[v % 80] + 1 + v // 80) & 3
            parts += [x for _ in range(copies) for x in (u, rng.integers(0, 4, 7))]
    g = np.concatenate(parts).astype(np.uint8)
    reads = [r.astype(np.uint8) for r in reads] + [(3 - r.astype(np.uint8))[::-1].copy() for r in reads]
    fm = oracle.FMIndex(g)
    for full_sa in (True, False):
        idx = gc.mica().Index.build(synth.to_acgt_bytes(g), kmer_q=12, sa_sample=8, full_sa=full_sa)
        for k in (0, 1):
            b = gc.batch_from_reads(reads, [k] * len(reads))
            gc.assert_same(idx.align_batch(b, hit_cap=cap), fm.align(b, cap=cap), f"cap {cap} k {k} full {full_sa}")
        idx.free()


@pytest.mark.parametrize("kmer_q", [1, 4, 8, 11])
def test_seeds_too_short_to_be_checked(kmer_q):
    """An index whose seeds are shorter than the text check asks for searches by
    the sweep and the trees too: every interval is checked once enough bases
    are matched."""
    _, a, _, want = _inputs()
    idx = gc.mica().Index.build(synth.to_acgt_bytes(_inputs()[0]), kmer_q=kmer_q, sa_sample=8)
    for cap in (20, 0):
        gc.assert_same(idx.align_batch(a, hit_cap=cap), want[cap], f"q {kmer_q} cap {cap}")
    assert idx.stats()["verified"] > 0
    if kmer_q > 4:
        _path_is_the_trees(idx)
    idx.free()


@pytest.mark.parametrize("verify", [1, 13, 20, 60, 255])
def test_a_verify_threshold_past_the_seeds(verify):
    """bidir_verify above the seeds' length leaves the sweep and the trees in place."""
    _, a, _, want = _inputs()
    idx = _index()
    idx.set_tuning(bidir_verify=verify)
    gc.assert_same(idx.align_batch(a, hit_cap=20), want[20], f"verify {verify}")
    _path_is_the_trees(idx)
    idx.free()


def test_captured_rounds_fall_again_after_a_hard_batch():
    """A batch that needs many rounds makes the workspace's captured batches hold as
    many; batches that need few bring them down again."""
    _, a, b, want = _inputs()
    idx = _index()
    easy = a.subset(np.arange(40))
    fm = oracle.FMIndex(_inputs()[0]).align(easy, cap=20)
    for _ in range(2):
        gc.assert_same(idx.align_batch(easy, hit_cap=20), fm, "before")
    few = idx.stats()["launches"]
    idx.debug_search_limits(steps=1)
    for _ in range(2):
        gc.assert_same(idx.align_batch(a, hit_cap=20), want[20], "hard")
    idx.debug_search_limits()
    gc.assert_same(idx.align_batch(easy, hit_cap=20), fm, "after")
    assert idx.stats()["launches"] > few
    for _ in range(40):
        gc.assert_same(idx.align_batch(easy, hit_cap=20), fm, "later")
    assert idx.stats()["launches"] == few and idx.stats()["graph_replays"] == 1
    idx.free()


@pytest.mark.parametrize("full_sa", [True, False])
def test_the_pool_gives_no_read_up_for_room(full_sa):
    """Pieces of six and seven bases, k = 3: the trees stop almost at once, and the
    warp pool searches nearly everything without handing on more nodes than the
    frontier holds."""
    g = synth.uniform_genome(600_000, 4)
    rng = np.random.default_rng(13)
    n = 205_000
    b = synth.sample_reads(g, np.full(n, 25), np.full(n, 3), rng, subs="rate", sub_rate=0.01)
    idx = gc.mica().Index.build(synth.to_acgt_bytes(g.codes), full_sa=full_sa)
    want = idx.align_batch(b, hit_cap=10, kernel="persistent")
    for call in range(2):
        gc.assert_same(idx.align_batch(b, hit_cap=10), want, f"call {call}")
        assert idx.stats()["warp_rounds"] > 0 and idx.stats()["fallback_reads"] == 0
    idx.free()

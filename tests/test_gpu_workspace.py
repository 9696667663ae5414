"""Device memory that a call's workspace takes, against what the library reports,
and what a workspace keeps between calls."""
import numpy as np
import pytest

import synth
from tests import gpu_common as gc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", ["plain", "short"])
def test_reported_workspace_covers_what_a_tick_reserves(batch):
    """A worker's tick takes no more device memory than
    mica_server_workspace_bytes reports for it, with the trees alone and with the
    warp pool (short reads): measured on the device, with a granule per buffer."""
    import torch
    m = gc.mica()
    g = synth.genome_64m(1 << 22)
    rng = np.random.default_rng(3)
    n, lens = 600_000, {"plain": 100, "short": 30}[batch]
    b = synth.sample_reads(g, np.full(n, lens), np.full(n, 2), rng, subs="rate", sub_rate=0.01)
    few = b.subset(np.arange(1_000))
    idx = m.Index.build(synth.to_acgt_bytes(g.codes))
    with m.Server(idx, workers=1, hit_cap=1) as srv:          # everything the process allocates once
        srv.wait(srv.submit_batch(few))
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    with m.Server(idx, workers=1, hit_cap=1, max_tick_reads=n, chunk_reads=n) as srv:
        srv.wait(srv.submit_batch(b))
        assert srv.stats()["ticks"] == 1
        used = before - torch.cuda.mem_get_info()[0]
        assert srv.stats()["device_bytes_in_use"] == m.Server.workspace_bytes(idx, n, int(b.word_off[-1]))
    assert used <= m.Server.workspace_bytes(idx, n, int(b.word_off[-1])) + (64 << 20)
    idx.free()


def test_other_kernels_are_charged_for_their_own_buffers():
    """A budget that holds the persistent kernel's tick but not the default
    kernel's is enough for a server of the former."""
    idx = gc.gpu_index("64m")
    m = gc.mica()
    b = synth.reads_64m(gc.genome("64m"), n=500)
    share = m.Server.workspace_bytes(idx, 500, 500 * 16) - (100 << 20)
    with m.Server(idx, workers=1, max_device_bytes=share) as srv:
        with pytest.raises(m.MicaError) as e:
            srv.submit_batch(b)
        assert e.value.code == m.MICA_ENOMEM
    with m.Server(idx, workers=1, max_device_bytes=share, kernel="persistent") as srv:
        res, _ = srv.wait(srv.submit_batch(b))
        gc.assert_same(res, idx.align_batch(b, hit_cap=1000))


@pytest.mark.parametrize("n", [16384 * 512, 16384 * 512 + 1, 16384 * 512 + 513])
def test_batches_around_the_most_tiles_every_block_adds_up(n):
    """The prefix sums of a batch of 8.4M reads, at the size from which a kernel
    scans the tiles' sums: totals, offsets and hits are those of the same reads
    in batches of a million."""
    import torch
    m = gc.mica()
    g = synth.uniform_genome(1 << 16, 2)
    idx = m.Index.build(synth.to_acgt_bytes(g.codes), kmer_q=8)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    dev = {"device": "cuda"}
    at = torch.randint(0, g.n - 16, (n,), generator=gen, **dev)
    codes = torch.from_numpy(g.codes).cuda().long()
    words = torch.zeros(n, dtype=torch.int64, **dev)
    for i in range(16):
        words |= codes[at + i] << (2 * i)
    words = torch.where(torch.rand(n, generator=gen, **dev) < 0.1, words ^ 7, words)   # some that do not occur
    words = torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32)
    off = torch.arange(n + 1, dtype=torch.int64, **dev)
    lens, k = torch.full((n,), 16, dtype=torch.int16, **dev), torch.zeros(n, dtype=torch.uint8, **dev)
    t, o, h = (x.clone() for x in idx.align_device(words, off, lens, k, n, hit_cap=3).tensors())
    o, h = o.view(torch.int64), h.view(torch.int64)
    assert int(o[0]) == 0 and int(o[-1]) == h.shape[0]
    at0 = 0
    for a in range(0, n, 1_000_000):
        c = min(1_000_000, n - a)
        ts, os_, hs = idx.align_device(words[a:a + c].clone(), off[:c + 1], lens[:c], k[:c], c, hit_cap=3).tensors()
        hs = hs.view(torch.int64)
        assert torch.equal(t[a:a + c], ts)
        assert torch.equal(o[a:a + c + 1] - at0, os_.view(torch.int64))
        assert torch.equal(h[at0:at0 + hs.shape[0]], hs)
        at0 += int(hs.shape[0])
    assert at0 == h.shape[0]
    idx.free()


@pytest.mark.parametrize("full_sa", [True, False])
def test_device_bytes_of_an_index(full_sa):
    """Index.device_bytes() is what the index takes on the device (up to a granule
    per array), the rows' left contexts included."""
    import torch
    m = gc.mica()
    g = synth.uniform_genome(20_000_000, 6)
    m.Index.build(synth.to_acgt_bytes(g.codes[:100_000])).free()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    idx = m.Index.build(synth.to_acgt_bytes(g.codes), full_sa=full_sa)
    used = before - torch.cuda.mem_get_info()[0]
    info = idx.info()
    listed = sum(info[x] for x in ("occ_bytes", "mark_bytes", "sample_bytes", "table_bytes", "rev_occ_bytes", "rev_table_bytes",
                                   "full_sa_bytes", "long_table_bytes"))
    assert idx.device_bytes() >= listed + (4 * (g.n + 1) if full_sa else 0)
    assert abs(used - idx.device_bytes()) <= 14 * (2 << 20)
    idx.free()


def test_every_table_lookup_is_counted():
    """stats()["seeds"]: a lookup per piece and strand, and another in the reversed
    genome's table for each seed that becomes a tree (the sweep) or for all (the
    warp pool)."""
    g = synth.uniform_genome(50_000, 12)
    rng = np.random.default_rng(1)
    n = 1_000
    b = synth.sample_reads(g, np.full(n, 60), np.full(n, 1), rng, subs="count", max_subs=0)
    idx = gc.mica().Index.build(synth.to_acgt_bytes(g.codes), kmer_q=10, sa_sample=8, full_sa=False)
    idx.align_batch(b)
    assert 4 * n + 2 * n <= idx.stats()["seeds"] <= 8 * n     # both pieces of the read's own strand occur
    idx.set_tuning(bidir_budget=16)
    idx.align_batch(b)
    assert idx.stats()["seeds"] == 8 * n
    idx.free()


def test_autotune_keeps_the_pools_defaults_where_the_trees_search():
    """Where no shape or budget of the warp pool reaches a kernel the autotuner does
    not choose among them, whatever was set before; where the pool searches
    (an index whose text check is off) it does."""
    g = synth.uniform_genome(200_000, 3)
    rng = np.random.default_rng(8)
    b = synth.sample_reads(g, np.full(2_000, 100), np.full(2_000, 2), rng, subs="rate", sub_rate=0.01)
    idx = gc.mica().Index.build(synth.to_acgt_bytes(g.codes))
    for shape in (0, 1):
        idx.set_tuning(bidir_shape=shape, bidir_budget=1024)
        for _ in range(3):
            t = idx.autotune(b, repeats=1)
            assert (t["bidir_shape"], t["bidir_budget"]) == (0, 4096)
    idx.set_tuning(bidir_verify=256)
    t = idx.autotune(b, repeats=1)
    assert t["bidir_shape"] in (0, 1) and t["bidir_budget"] in (1024, 4096) and t["bidir_verify"] == 256
    idx.free()

"""What users have this library do, as cases that can be timed: searches of
read batches against a resident index, from a handful of probes to a million
reads, with reads and results on the device or on the host, one call at a time,
pipelined or through the server, and the construction of an index.

A case is a dict of plain values:

  way      how the call is made: "device" (reads and results in device memory), "host" (host arrays in and
           out), "pairs" (device, then mate pairing), "stream" (pinned host batches, two in flight), "serve"
           (requests through the server) or "build" (a new index, then its first batch)
  genome   "random" (i.i.d. bases), "repeats" (1-10 kbp copies at 1% divergence over 5%, exact tandem arrays over
           1%) or "human" (300 bp families at 10-15% divergence over 15%, 6 kbp families at 5% over 25%, tandem
           arrays at 1-5% over 5%), of `bases` bases
  reads    reads per batch (per pass for "serve"), with lengths lo..hi ("few": only 100, 150 and 250 of them),
           budget k (kmax: each read draws 0..kmax) and errors at 1% per base; `inside` of them start in a repeat
  cap      hits listed per read;  report  "all" or "best_stratum";  full  whether the index keeps the whole
           suffix array and the text
"""
import math

import numpy as np
import torch

import paper_1402_4876_gb300 as mica

_BASE = {"way": "device", "genome": "repeats", "bases": 1 << 26, "reads": 1000, "lo": 150, "hi": 150, "few": False,
         "k": 2, "mixed_k": False, "inside": 0.0, "cap": 1000, "report": "all", "full": True}


def _case(**kw):
    return {**_BASE, **kw}


def listed():
    return [
        # a few probes looked up interactively: the smallest call, all latency
        _case(name="probes_64", way="host", genome="random", bases=1_000_000, reads=64, lo=100, hi=100),
        # the small workload: a 1 Mbp genome (a bacterium, a panel), ten thousand 100 bp reads from host arrays
        _case(name="panel_10k", way="host", genome="random", bases=1_000_000, reads=10_000, lo=100, hi=100),
        # the headline: a 64 Mbp genome with repeats, a million 150 bp reads resident on the device
        _case(name="repeats_1m", reads=1_000_000),
        # uneven batches: lengths 50..250, budgets 0..3, 30% of the reads inside repeats (the heavy tail)
        _case(name="uneven_1m", reads=1_000_000, lo=50, hi=250, k=3, mixed_k=True, inside=0.3),
        # paired-end resequencing against a genome whose index lives in HBM: search of both mates, then pairing
        _case(name="human_pairs", way="pairs", genome="human", bases=1 << 29, reads=1_000_000),
        # a lane streamed from pinned host memory: batches of 250k reads, two in flight
        _case(name="stream_4x250k", way="stream", reads=250_000),
        # long reads with the largest budget, only the best placements wanted, ordinary host arrays
        _case(name="best_long", way="host", bases=1 << 24, reads=100_003, lo=250, hi=250, k=3, report="best_stratum"),
        # short odd-length reads (small RNA, ChIP tags) with a low cap
        _case(name="short_odd", bases=1 << 23, reads=33_333, lo=36, hi=75, k=1, mixed_k=True, inside=0.2, cap=10),
        # an index without the suffix array and text (small memory): base-by-base extension, LF-walk locate
        _case(name="lean_index", bases=1 << 24, reads=50_000, lo=100, hi=100, full=False),
        # requests of mixed sizes, lengths and budgets through the continuous-batching server
        _case(name="serve_mix", way="serve", genome="human", bases=1 << 25, reads=400_000, lo=100, hi=250, few=True,
              mixed_k=True),
        # a new reference: its index is built and the first reads are placed
        _case(name="build_16m", way="build", genome="human", bases=1 << 24, reads=2_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    way = rng.choice(["host", "device", "device", "pairs", "stream", "serve", "build", "lean"])
    lo = rng.randint(36, 250)
    hi = rng.choice([lo, rng.randint(lo, 250)])
    k = rng.randint(0, min(3, lo // 30))
    c = {"genome": rng.choice(["random", "repeats", "human"]), "bases": _log(rng, 1 << 20, 1 << 26),
         "reads": _log(rng, 50, 400_000), "lo": lo, "hi": hi, "k": k, "mixed_k": rng.random() < 0.4,
         "inside": rng.choice([0.0, 0.0, 0.2]), "cap": rng.choice([1, 10, 1000, 1000]),
         "report": rng.choice(["all", "all", "all", "best_stratum"])}
    if way in ("host", "stream"):
        c["inside"] = 0.0
    if way == "lean":
        c.update(full=False, bases=_log(rng, 1 << 20, 1 << 24), reads=_log(rng, 50, 40_000), lo=max(lo, 60),
                 hi=max(hi, 60), k=min(k, 2), genome=rng.choice(["random", "repeats"]))
        way = "device"
    elif way == "pairs":
        c.update(genome="human", bases=_log(rng, 1 << 23, 1 << 28), reads=2 * _log(rng, 50, 150_000),
                 lo=rng.choice([100, 150]), k=2, mixed_k=False, inside=0.0, report="all", cap=1000)
        c["hi"] = c["lo"]
    elif way == "serve":
        c.update(reads=_log(rng, 2_000, 300_000), few=True, lo=100, hi=250, k=2, mixed_k=True, inside=0.0,
                 report="all", cap=1000)
    elif way == "build":
        c.update(bases=_log(rng, 1 << 20, 1 << 24), reads=_log(rng, 50, 2_000))
    elif way == "stream":
        c.update(reads=_log(rng, 1_000, 200_000))
    return _case(way=way, **c)


# ---- genomes: uint8 base codes on the device, planted repeats as (starts, lengths) ----

def _cells(g, n, count, size, lens, gen):
    """Distinct places for `count` stretches of `lens` <= `size` bases: one per cell, so none overlap."""
    cells = n // size
    count = min(count, cells)
    at = torch.randperm(cells, generator=gen, device=g.device)[:count] * size
    lens = lens[:count]
    return at + (torch.rand(count, generator=gen, device=g.device) * (size - lens + 1)).long(), lens


def _plant(g, starts, lens, source, div, gen):
    """Write source(rows, t) at starts + t for t < lens, each base substituted with its row's probability `div`."""
    if starts.numel() == 0:
        return
    width = int(lens.max())
    step = max(1, (1 << 24) // width)
    t = torch.arange(width, device=g.device)
    for r0 in range(0, starts.numel(), step):
        rows = torch.arange(r0, min(starts.numel(), r0 + step), device=g.device)
        v = source(rows, t)
        hit = torch.rand(v.shape, generator=gen, device=g.device) < div[rows][:, None]
        shift = torch.randint(1, 4, v.shape, generator=gen, device=g.device, dtype=torch.uint8)
        v = torch.where(hit, (v + shift) & 3, v)
        keep = t[None, :] < lens[rows][:, None]
        g[(starts[rows][:, None] + t[None, :])[keep]] = v[keep]


def _oriented(v, rev):
    return torch.where(rev[:, None], 3 - v.flip(1), v)


def _genome(case, gen):
    n, dev = case["bases"], "cuda"
    g = torch.randint(0, 4, (n,), generator=gen, device=dev, dtype=torch.uint8)
    regions = []

    def rand(count, lo, hi):
        return torch.randint(lo, hi + 1, (count,), generator=gen, device=dev)

    def coin(count):
        return torch.rand(count, generator=gen, device=dev) < 0.5

    def tandem(frac, longest, d0, d1):
        c = max(1, int(frac * n / (longest / 2)))
        st, ln = _cells(g, n, c, longest, rand(c, 100, longest), gen)
        units = torch.randint(0, 4, (st.numel(), 50), generator=gen, device=dev, dtype=torch.uint8)
        u = rand(st.numel(), 2, 50)
        div = d0 + (d1 - d0) * torch.rand(st.numel(), generator=gen, device=dev)
        _plant(g, st, ln, lambda r, t: units[r].gather(1, t[None, :] % u[r][:, None]), div, gen)
        regions.append((st, ln))

    if case["genome"] == "repeats":
        c = max(1, int(0.05 * n / 5500))
        st, ln = _cells(g, n, c, 10_000, rand(c, 1000, 10_000), gen)
        src = (torch.rand(st.numel(), generator=gen, device=dev) * (n - 10_000)).long()
        rev, old = coin(st.numel()), g.clone()
        _plant(g, st, ln, lambda r, t: _oriented(old[src[r][:, None] + t[None, :]], rev[r]),
               torch.full((st.numel(),), 0.01, device=dev), gen)
        regions.append((st, ln))
        tandem(0.01, 5000, 0.0, 0.0)
    elif case["genome"] == "human":
        fam = torch.randint(0, 4, (50, 300), generator=gen, device=dev, dtype=torch.uint8)
        c = max(1, int(0.15 * n / 300))
        st, ln = _cells(g, n, c, 400, torch.full((c,), 300, device=dev), gen)
        f, rev = rand(st.numel(), 0, 49), coin(st.numel())
        _plant(g, st, ln, lambda r, t: _oriented(fam[f[r]], rev[r]),
               0.10 + 0.05 * torch.rand(st.numel(), generator=gen, device=dev), gen)
        regions.append((st, ln))
        fam6 = torch.randint(0, 4, (20, 6000), generator=gen, device=dev, dtype=torch.uint8)
        c = max(1, int(0.25 * n / 4575))
        ln = torch.where(coin(c), torch.full((c,), 6000, device=dev), rand(c, 300, 6000))
        st, ln = _cells(g, n, c, 6000, ln, gen)
        f6, rev6 = rand(st.numel(), 0, 19), coin(st.numel())

        def copy6(r, t):
            # a 5'-truncated copy keeps its consensus's 3' end; a reversed one is its other strand
            i = torch.where(rev6[r][:, None], 5999 - t[None, :], (6000 - ln[r])[:, None] + t[None, :]).clamp(max=5999)
            v = fam6[f6[r]].gather(1, i)
            return torch.where(rev6[r][:, None], 3 - v, v)

        _plant(g, st, ln, copy6, torch.full((st.numel(),), 0.05, device=dev), gen)
        regions.append((st, ln))
        tandem(0.05, 20_000, 0.01, 0.05)
    if not regions:
        return g, None
    return g, (torch.cat([a for a, _ in regions]), torch.cat([b for _, b in regions]))


# ---- reads: 2-bit packed, 16 bases per word, least significant first ----

def _pack(mat, lens):
    """Rows of base codes -> (words int32, word offsets int64)."""
    nw = (lens + 15) // 16
    off = torch.zeros(lens.numel() + 1, dtype=torch.int64, device=mat.device)
    torch.cumsum(nw, 0, out=off[1:])
    wide, parts = (mat.shape[1] + 15) // 16, []
    sh = 2 * torch.arange(16, device=mat.device)
    for r0 in range(0, mat.shape[0], 1 << 18):
        m = mat[r0:r0 + (1 << 18)]
        m = torch.where(torch.arange(m.shape[1], device=m.device)[None, :] < lens[r0:r0 + m.shape[0], None], m, 0)
        m = torch.nn.functional.pad(m, (0, wide * 16 - m.shape[1])).view(-1, wide, 16)
        w = torch.zeros(m.shape[:2], dtype=torch.int64, device=m.device)
        for i in range(16):
            w |= m[:, :, i].long() << sh[i]
        keep = torch.arange(wide, device=m.device)[None, :] < nw[r0:r0 + m.shape[0], None]
        parts.append(w[keep])
    words = torch.cat(parts) if parts else torch.zeros(0, dtype=torch.int64, device=mat.device)
    return torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32), off


def _mutate(mat, rate, gen):
    for r0 in range(0, mat.shape[0], 1 << 18):
        m = mat[r0:r0 + (1 << 18)]
        hit = torch.rand(m.shape, generator=gen, device=m.device) < rate
        shift = torch.randint(1, 4, m.shape, generator=gen, device=m.device, dtype=torch.uint8)
        m.copy_(torch.where(hit, (m + shift) & 3, m))


def _windows(g, start, lens, rev):
    """Rows g[start, start + len), the other strand where rev; past a row's length the bases are arbitrary."""
    out = torch.empty((start.numel(), int(lens.max())), dtype=torch.uint8, device=g.device)
    t = torch.arange(out.shape[1], device=g.device)
    for r0 in range(0, start.numel(), 1 << 18):
        s, ln, rv = (x[r0:r0 + (1 << 18), None] for x in (start, lens, rev))
        i = torch.where(rv, ln - 1 - t[None, :], t[None, :])
        v = g[(s + i).clamp(0, g.numel() - 1)]
        out[r0:r0 + s.shape[0]] = torch.where(rv, 3 - v, v)
    return out


def _reads(case, n, g, regions, gen):
    """(base codes, lengths, budgets) of n reads of the genome."""
    dev = g.device
    if case["few"]:
        some = torch.tensor([m for m in (100, 150, 250) if case["lo"] <= m <= case["hi"]], device=dev)
        lens = some[torch.randint(0, some.numel(), (n,), generator=gen, device=dev)]
    else:
        lens = torch.randint(case["lo"], case["hi"] + 1, (n,), generator=gen, device=dev)
    if case["way"] == "pairs":
        # mates 2i, 2i + 1 of a fragment: Normal(500, 50) clipped to 300..700, forward/reverse library; the
        # sequenced individual differs from the reference by 0.1%
        frag = (500 + 50 * torch.randn(n // 2, generator=gen, device=dev)).round().clamp(300, 700).long()
        a = (torch.rand(n // 2, generator=gen, device=dev) * (g.numel() - frag + 1)).long()
        first = torch.rand(n // 2, generator=gen, device=dev) < 0.5
        left, right = a, a + frag - case["lo"]
        start = torch.stack([torch.where(first, left, right), torch.where(first, right, left)], 1).view(-1)
        rev = torch.stack([~first, first], 1).view(-1)
    else:
        start = (torch.rand(n, generator=gen, device=dev) * (g.numel() - lens + 1)).long()
        if case["inside"] and regions is not None:
            st, ln = regions
            r = torch.multinomial(ln.double(), n, replacement=True, generator=gen)
            s = st[r] + (torch.rand(n, generator=gen, device=dev) * (ln[r] - lens + 1).clamp(min=1)).long()
            pick = torch.rand(n, generator=gen, device=dev) < case["inside"]
            start = torch.where(pick, torch.minimum(s, g.numel() - lens), start)
        rev = torch.rand(n, generator=gen, device=dev) < 0.5
    mat = _windows(g, start, lens, rev)
    _mutate(mat, 0.011 if case["way"] == "pairs" else 0.01, gen)
    k = torch.full((n,), case["k"], device=dev, dtype=torch.uint8)
    if case["mixed_k"]:
        k = torch.randint(0, case["k"] + 1, (n,), generator=gen, device=dev).to(torch.uint8)
    return mat, lens, k


def _batches(case):
    """Reads of each batch of a pass."""
    if case["way"] == "stream":
        return [case["reads"]] * 4
    if case["way"] == "serve":
        # ten requests whose sizes span a factor of a hundred
        w = [100 ** (-i / 9) for i in range(10)]
        return [max(1, int(case["reads"] * x / sum(w))) for x in w]
    return [case["reads"]]


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    g, regions = _genome(case, gen)
    return g, [_reads(case, n, g, regions, gen) for n in _batches(case)]


class _State(dict):
    """What a pass needs; its server and index go in that order."""

    def __del__(self):
        if self.get("server") is not None:
            self["server"].stop()
        if self.get("index") is not None:
            self["index"].free()


def _room(case, n):
    """Length of the program's own hit array for a batch of n reads (-1 past the hits listed)."""
    return n * min(case["cap"], 160 if case["way"] in ("device", "pairs") else 64) + (1 << 16)


def prepare(case, seed):
    case = {**_BASE, **case}
    g, batches = _inputs(case, seed)
    acgt = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device=g.device)
    text = acgt[g.long()].cpu().numpy() if g.numel() <= 1 << 27 else np.concatenate(
        [acgt[p.long()].cpu().numpy() for p in g.split(1 << 27)])
    del g
    device = case["way"] in ("device", "pairs")
    s = _State(case=case, index=None, server=None, batches=[], hits=[])
    for mat, lens, k in batches:
        words, off = _pack(mat, lens)
        arrays = (words, off, lens.to(torch.int16), k)
        if not device:
            arrays = [x.cpu() for x in arrays]
            if case["way"] == "stream":
                arrays = [x.pin_memory() for x in arrays]
            s.setdefault("held", []).append(arrays)
            arrays = [x.numpy().view(t) for x, t in zip(arrays, (np.uint32, np.uint64, np.uint16, np.uint8))]
        s["batches"].append(tuple(arrays))
        s["hits"].append(torch.full((_room(case, lens.numel()),), -1, dtype=torch.int64, device="cuda" if device else "cpu"))
    del batches, mat, lens, k
    torch.cuda.empty_cache()
    if case["way"] == "build":
        s["text"] = text
        return s
    s["index"] = mica.Index.build(text, full_sa=case["full"])
    if case["way"] == "serve":
        s["server"] = mica.Server(s["index"], hit_cap=case["cap"])
    if case["way"] == "pairs":
        s["paired"] = torch.zeros(case["reads"] // 2 * mica.PAIR_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    return s


def _host(res, mine):
    if res.hits.size:
        mine[:res.hits.size].copy_(torch.from_numpy(res.hits.view(np.int64)))
    return [res.total.view(np.int64), res.offsets.view(np.int64), mine]


def run(state):
    c, idx, batches, mine = state["case"], state["index"], state["batches"], state["hits"]
    opts = {"hit_cap": c["cap"], "report": c["report"]}
    if c["way"] == "host":
        return _host(idx.align(*batches[0], **opts), mine[0])
    if c["way"] in ("device", "pairs"):
        b = batches[0]
        res = idx.align_device(*b, c["reads"], **opts)
        total, offsets, hits = res.tensors()
        mine[0][:res.n_hits].copy_(hits.view(torch.int64))
        out = [total.view(torch.int64), offsets.view(torch.int64), mine[0]]
        for x in out[:2]:
            x.owner = state   # views of the index's memory, which lives while they do
        if c["way"] == "pairs":
            mica.pair_device(offsets, hits, b[2], c["reads"] // 2, 300, 700, state["paired"])
            out.append(state["paired"])
        return out
    if c["way"] == "stream":
        out, before = [], None
        for b in batches:
            ticket = idx.submit(*b, **opts)
            if before is not None:
                out.append(_host(idx.collect(before), mine[len(out)]))
            before = ticket
        out.append(_host(idx.collect(before), mine[len(out)]))
        return out
    if c["way"] == "serve":
        rids = [state["server"].submit(*b) for b in batches]
        return [_host(state["server"].wait(r)[0], m) for r, m in zip(rids, mine)]
    new = mica.Index.build(state["text"], full_sa=c["full"])
    out = _host(new.align(*batches[0], **opts), mine[0])
    new.free()
    return out


def work(case):
    """Least bytes of a pass: the packed reads, offsets, lengths and budgets in; total, offset and one placement
    per read out; one table entry pair for each of a read's k + 1 pieces on both strands; for the placement, its
    suffix array entry and the text under it.  A new index adds its text in and its occurrence blocks, suffix
    array, inverse and text out.  No floating-point work: everything is integer."""
    c = {**_BASE, **case}
    n = sum(_batches(c))
    m, k = (c["lo"] + c["hi"]) / 2, c["k"] / 2 if c["mixed_k"] else c["k"]
    nbytes = n * (4 * math.ceil(m / 16) + 11 + 24 + 2 * (k + 1) * 8 + 4 + m / 4)
    if c["way"] == "pairs":
        nbytes += n // 2 * mica.PAIR_DTYPE.itemsize
    if c["way"] == "build":
        nbytes += c["bases"] * (1 + 2 / 3 + 8 + 0.25)
    return {"bytes": nbytes, "flops": 0}


def exact(case, seed):
    """The placements by pigeonhole, in 64-bit integers: some piece of a read with at most k substitutions is
    exact, so every occurrence of each piece's first bases is a candidate, and each candidate window is compared
    base by base.  Listed hits only where no read is over its cap (the cap's order follows the suffix array)."""
    c = {**_BASE, **case}
    n = c["bases"]
    if c["genome"] != "random" or n > 1 << 24 or c["way"] not in ("host", "device") or c["lo"] < 16 * (c["k"] + 1):
        return None
    g, [(mat, lens, budget)] = _inputs(c, seed)
    p = c["k"] + 1
    q = min(20, c["lo"] // p)
    if n * 0.5 ** (2 * q) * c["reads"] * p > 1e8:
        return None
    code = torch.zeros(n - q + 1, dtype=torch.int64, device=g.device)
    for t in range(q):
        code = code * 4 + g[t:n - q + 1 + t]
    code, place = torch.sort(code)
    ids = torch.arange(mat.shape[0], device=g.device)
    zeros = torch.zeros_like(ids)
    found = []
    for strand in (0, 1):
        pat = mat
        if strand:
            i = (lens[:, None] - 1 - torch.arange(mat.shape[1], device=g.device)[None, :]).clamp(min=0)
            pat = 3 - mat.gather(1, i)
        for piece in range(p):
            a = zeros + piece * lens // p
            key = zeros
            for t in range(q):
                key = key * 4 + pat.gather(1, (a + t)[:, None])[:, 0]
            first, last = torch.searchsorted(code, key), torch.searchsorted(code, key, right=True)
            count = last - first
            read = ids.repeat_interleave(count)
            nth = torch.arange(read.numel(), device=g.device) - (count.cumsum(0) - count)[read]
            start = place[first[read] + nth] - a[read]
            for j in range(0, read.numel(), 1 << 20):
                r, s = read[j:j + (1 << 20)], start[j:j + (1 << 20)]
                ok = (s >= 0) & (s + lens[r] <= n)
                r, s = r[ok], s[ok]
                t = torch.arange(pat.shape[1], device=g.device)[None, :]
                differ = g[(s[:, None] + t).clamp(max=n - 1)] != pat[r]
                d = (differ & (t < lens[r][:, None])).sum(1)
                ok = d <= budget[r]
                found.append(((r[ok] * n + s[ok]) * 2 + strand) * 4 + d[ok])
    hit = torch.unique(torch.cat(found))
    d, strand, pos, read = hit % 4, hit // 4 % 2, hit // 8 % n, hit // 8 // n
    if c["report"] == "best_stratum":
        best = torch.full_like(ids, 4).scatter_reduce(0, read, d, "amin")
        keep = d == best[read]
        d, strand, pos, read = d[keep], strand[keep], pos[keep], read[keep]
    total = torch.bincount(read, minlength=ids.numel())
    offsets = torch.cat([zeros[:1], total.clamp(max=c["cap"]).cumsum(0)])
    hits = None
    if int(total.max()) <= c["cap"]:
        hits = torch.full((_room(c, ids.numel()),), -1, dtype=torch.int64, device=g.device)
        hits[:pos.numel()] = pos | strand << 32 | d << 40
    return [total, offsets, hits]

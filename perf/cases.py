"""The work whose speed is measured: countBF counting through the public API.

Every case is one call pattern of a program that uses the library:

  count    reads resident on the device: reset, insert, classify, and the
           countBF cells and both key lists taken out;
  job      the same for one job of a counting service: reads in pinned host
           memory, results and totals back on the host;
  stream   one sample that arrives in several pieces from pinned host
           memory, each inserted as it comes, classified at the end;
  batch    many samples of uneven size counted together (Batch);
  merge    two counted shards merged into one handle and classified;
  query    frequency queries of a countBF that is already filled.

Reads are sampled from a random genome (uniform or GC-poor, optionally with
repeat families) on both strands with substitution errors and N calls.  All
outputs are whole numbers.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2305_07545_gb300 as kc

_ACGT = (65, 67, 71, 84)


def _case(name: str | None, kind: str, **kw) -> dict:
    c = dict(kind=kind, K=31, reads=0, len_lo=150, len_hi=150, genome=1_000_000, gc=0.5, sub=0.01,
             n_rate=0.0, repeats=False, m=1 << 20, eq1=False, alpha=4, nhash=4, tau=3, pieces=1,
             samples=1, keys=0)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed() -> list[dict]:
    return [
        # a small amplicon or plasmid sample: launch and latency bound
        _case("tiny", "count", K=21, reads=2_000, len_lo=100, len_hi=100, genome=50_000,
              n_rate=0.001, m=1 << 20, nhash=3, tau=2),
        # the smallest job of the counting service's size distribution, host to host
        _case("job", "job", reads=10_007, len_lo=50, len_hi=300, genome=1_000_000,
              m=8 * 1_100_003 // 4),
        # one bacterial genome at 30x
        _case("single", "count", reads=1_000_000, genome=5_000_000, gc=0.41, sub=0.005, m=1 << 28),
        # the paper's setting: Eq. 1 prime dimensions, 8-bit counters, both of its K
        _case("paper28", "count", K=28, reads=1_000_000, genome=5_000_000, gc=0.41, sub=0.005,
              eq1=True, alpha=8, nhash=3, tau=5),
        _case("paper55", "count", K=55, reads=700_001, genome=5_000_000, gc=0.41, sub=0.005,
              eq1=True, alpha=8, nhash=3, tau=5),
        # a large repetitive genome, one-word and two-word keys, 4 GiB countBF
        _case("repeats", "count", reads=6_000_000, genome=30_000_000, repeats=True, m=1 << 33),
        _case("repeats55", "count", K=55, reads=4_000_000, genome=20_000_000, repeats=True,
              m=1 << 33),
        # a countBF tuned for few false positives (seven hashes), ragged reads with N calls,
        # a counter number that is no power of two
        _case("hashes7", "count", K=25, reads=300_007, len_lo=50, len_hi=300, genome=3_000_017,
              n_rate=0.001, m=200_000_003, alpha=8, nhash=7, tau=4),
        # sixteen samples of log-normal size under one graph
        _case("batch", "batch", samples=16, reads=140_000, len_lo=50, len_hi=300,
              genome=1_000_000),
        # a sample that arrives in pieces
        _case("stream", "stream", reads=800_003, pieces=16, genome=4_000_000, sub=0.005,
              m=1 << 27),
        # two shards of one sample brought together
        _case("merge", "merge", reads=600_000, genome=4_000_000, sub=0.005, m=1 << 27),
        # frequency queries, half of the keys present
        _case("query", "query", reads=500_000, genome=4_000_000, sub=0.005, m=1 << 28,
              keys=10_000_019),
    ]


def _logint(rng: random.Random, lo: float, hi: float) -> int:
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng: random.Random) -> dict:
    kind = rng.choice(["count"] * 6 + ["job", "stream", "batch", "merge", "query"])
    K = rng.choice([15, 17, 21, 21, 23, 25, 27, 28, 31, 31, 31, 32, 33, 41, 51, 55, 55, 63])
    alpha = rng.choice([4, 4, 4, 8, 8, 5, 6, 12, 16])
    nhash = rng.choice([2, 3, 3, 4, 4, 4, 5, 7])
    lo, hi = rng.choice([(100, 100), (150, 150), (151, 151), (50, 300), (100, 250)])
    most = {"count": 5e6 if K <= 32 else 3e6, "job": 4e5, "stream": 1e6, "batch": 1.6e5,
            "merge": 8e5, "query": 8e5}[kind]
    if nhash > 4:
        most = min(most, 3e5)
    if hi > 151:
        most *= 0.75
    reads = _logint(rng, {"batch": 2e4}.get(kind, 2e3), most)
    windows = max(1, reads * ((lo + hi) // 2 - K + 1))
    eq1 = rng.random() < 0.25
    m = min(1 << 33, max(1 << 18, int(windows * math.exp(rng.uniform(math.log(2), math.log(12))))))
    if rng.random() < 0.5:
        m = 1 << (m.bit_length() - 1)
    return _case(None, kind, K=K, reads=reads, len_lo=lo, len_hi=hi,
                 genome=max(20_000, int(reads * (lo + hi) / 2 / rng.uniform(8, 40))),
                 gc=rng.choice([0.5, 0.41, 0.35]), sub=rng.choice([0.002, 0.005, 0.01, 0.02]),
                 n_rate=rng.choice([0.0, 0.0, 0.001]), repeats=rng.random() < 0.3, m=m, eq1=eq1,
                 alpha=alpha, nhash=nhash, tau=rng.choice([1, 2, 3, 5]),
                 pieces=rng.randint(2, 24) if kind == "stream" else 1,
                 samples=rng.randint(3, 16) if kind == "batch" else 1,
                 keys=_logint(rng, 1e3, 2e7) if kind == "query" else 0)


# ------------------------------------------------------------------ inputs
def _genome(c: dict, g: torch.Generator, seed: int) -> torch.Tensor:
    """Base indices 0..3 (A, C, G, T); with repeats a tenth of the genome is
    overwritten by diverged copies of a few families."""
    u = torch.rand(c["genome"], generator=g, device="cuda")
    at = (1.0 - c["gc"]) / 2
    codes = ((u >= at).to(torch.uint8) + (u >= at + c["gc"] / 2) + (u >= at + c["gc"]))
    if c["repeats"]:
        r = random.Random(seed)
        left = c["genome"] // 10
        while left > 0:
            flen = min(r.randint(500, 5000), c["genome"] // 4)
            fam = torch.randint(4, (flen,), generator=g, device="cuda", dtype=torch.uint8)
            copies = min(r.randint(2, 200), 1 + left // flen)
            div = torch.rand(copies, flen, generator=g, device="cuda") < 0.01
            many = torch.where(div, (fam + 1) & 3, fam)
            for i in range(copies):
                p = r.randrange(c["genome"] - flen)
                codes[p:p + flen] = many[i]
            left -= copies * flen
    return codes


def _reads(c: dict, seed: int, n: int | None = None) -> tuple[torch.Tensor, torch.Tensor]:
    """(bases uint8, offsets int64) of n reads on the device."""
    n = c["reads"] if n is None else n
    g = torch.Generator(device="cuda").manual_seed(seed)
    codes = _genome(c, g, seed)
    G = c["genome"]
    lens = torch.randint(c["len_lo"], c["len_hi"] + 1, (n,), generator=g, device="cuda")
    offsets = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=offsets[1:])
    ends = offsets[::1 << 18].tolist()
    total = int(offsets[-1])
    bases = torch.empty(total, dtype=torch.uint8, device="cuda")
    letters = torch.tensor(_ACGT, dtype=torch.uint8, device="cuda")
    for i, r0 in enumerate(range(0, n, 1 << 18)):
        r1 = min(n, r0 + (1 << 18))
        b0, b1 = ends[i], (ends[i + 1] if i + 1 < len(ends) and r1 < n else total)
        L, nb = lens[r0:r1], b1 - b0
        rid = torch.repeat_interleave(torch.arange(r1 - r0, device="cuda"), L, output_size=nb)
        pos = torch.arange(nb, device="cuda") - (offsets[r0:r1] - b0)[rid]
        rev = (torch.rand(r1 - r0, generator=g, device="cuda") < 0.5)[rid]
        start = torch.randint(G, (r1 - r0,), generator=g, device="cuda")[rid]
        pos = torch.where(rev, L[rid] - 1 - pos, pos)
        x = codes[(start + pos) % G]
        x = torch.where(rev, 3 - x, x)
        err = torch.rand(nb, generator=g, device="cuda") < c["sub"]
        step = torch.randint(1, 4, (nb,), generator=g, device="cuda", dtype=torch.uint8)
        x = torch.where(err, (x + step) & 3, x)
        a = letters[x.long()]
        if c["n_rate"]:
            a[torch.rand(nb, generator=g, device="cuda") < c["n_rate"]] = 78
        bases[b0:b1] = a
    return bases, offsets


def _windows(c: dict) -> int:
    return max(1, c["reads"] * max(1, (c["len_lo"] + c["len_hi"]) // 2 - c["K"] + 1))


def _filter(c: dict, m: int | None = None, stream: int | None = None) -> kc.CountBF:
    dims = kc.kmerco_paper_dims(max(1, _windows(c) // 2), 0.001) if c["eq1"] else None
    return kc.CountBF(c["K"], c["m"] if m is None else m, c["alpha"], c["nhash"], c["tau"],
                      dims=dims, stream=stream)


def _sample_sizes(c: dict) -> list[int]:
    """Read counts of a batch: log-normal around c["reads"], the same for every seed."""
    r = random.Random(c["samples"])
    return [min(2 * c["reads"], max(c["reads"] // 14, int(c["reads"] * math.exp(r.gauss(0, 1.2)))))
            for _ in range(c["samples"])]


class _BatchState(dict):
    """The batch goes before the handles that it groups."""

    def __del__(self):
        self["batch"].close()
        for f in self["filters"]:
            f.close()


def prepare(case: dict, seed: int) -> dict:
    c = case
    kind = c["kind"]
    if kind == "batch":
        stream = torch.cuda.Stream()
        sizes = _sample_sizes(c)
        data = [_reads(c, 1000 * seed + i, n) for i, n in enumerate(sizes)]
        mean = max(1, (c["len_lo"] + c["len_hi"]) // 2 - c["K"] + 1)
        # eight bits for each distinct K-mer that is expected
        filters = [_filter(dict(c, reads=n, eq1=False), max(64, _distinct(c, n * mean) * 8 // c["alpha"]),
                           stream.cuda_stream) for n in sizes]
        st = _BatchState(c=c, stream=stream, filters=filters, batch=kc.Batch(filters),
                         bases=[b for b, _ in data], offsets=[o for _, o in data])
    elif kind == "merge":
        half = dict(c, reads=c["reads"] // 2)
        st = dict(c=c, bf=_filter(c), shards=[])
        bases, offsets = _reads(c, seed)
        cut = half["reads"]
        at = int(offsets[cut])
        for b, o in ((bases[:at], offsets[:cut + 1]), (bases[at:], offsets[cut:] - at)):
            f = _filter(c)
            torch.cuda.synchronize()
            f.insert(b.clone(), o.clone())
            f.classify()
            st["shards"].append(f)
    elif kind == "query":
        st = dict(c=c, bf=_filter(c))
        bases, offsets = _reads(c, seed)
        torch.cuda.synchronize()
        st["bf"].insert(bases, offsets)
        st["bf"].classify()
        g = torch.Generator(device="cuda").manual_seed(seed + 1)
        kw, n = st["bf"].kw, c["keys"]
        have = torch.cat([t.view(-1, kw) for t in _lists(st["bf"])])
        low = torch.randint(-2 ** 63, 2 ** 63 - 1, (n, kw), generator=g, device="cuda")
        spare = (64 if kw == 1 else 128) - 2 * c["K"]
        if spare:   # keys of 2K bits
            low[:, kw - 1] = (low[:, kw - 1] >> spare) & ((1 << (64 - spare)) - 1)
        pick = torch.randint(len(have), (n,), generator=g, device="cuda")
        hit = torch.rand(n, generator=g, device="cuda") < 0.5
        st["keys"] = torch.where(hit[:, None], have[pick], low).contiguous()
    else:
        bases, offsets = _reads(c, seed)
        st = dict(c=c, bf=_filter(c))
        if kind == "count":
            st.update(bases=bases, offsets=offsets)
        elif kind == "job":
            st.update(bases=bases.cpu().pin_memory(), offsets=offsets.cpu().pin_memory())
        else:
            hb, ho = bases.cpu(), offsets.cpu()
            cuts = [c["reads"] * i // c["pieces"] for i in range(c["pieces"] + 1)]
            st["parts"] = [(hb[int(ho[a]):int(ho[b])].clone().pin_memory(),
                            (ho[a:b + 1] - ho[a]).clone().pin_memory())
                           for a, b in zip(cuts[:-1], cuts[1:]) if b > a]
    if kind == "batch":
        st["out"] = [_buffers(c, f, n * mean) for f, n in zip(filters, sizes)]
    elif kind != "query":
        st["out"] = _buffers(c, st["bf"], _windows(c), host=kind == "job")
    torch.cuda.synchronize()
    return st


# --------------------------------------------------------------------- run
def _lists(bf: kc.CountBF) -> list[torch.Tensor]:
    out = []
    for get in (kc.kmerco_get_trusted, kc.kmerco_get_erroneous):
        n = get(bf.h)
        keys = torch.empty(n * bf.kw, dtype=torch.int64, device="cuda")
        get(bf.h, keys, n)
        out.append(keys)
    return out


def _buffers(c: dict, bf: kc.CountBF, windows: int, host: bool = False) -> dict:
    """What a program keeps for the results of one handle: the cells and both
    lists, with room for the distinct K-mers that it expects."""
    words, cap = bf.stats()["words"], int(1.2 * _distinct(c, windows)) + 10_000
    sizes = (words, cap * bf.kw, cap * bf.kw)
    if host:
        bufs = [torch.zeros(n, dtype=torch.int64).pin_memory() for n in sizes]
    else:
        bufs = [torch.zeros(n, dtype=torch.int64, device="cuda") for n in sizes]
    return dict(words=words, cap=cap, bufs=bufs)


def _results(bf: kc.CountBF, r: dict) -> list:
    """The countBF cells and both key lists in the program's buffers, and the
    lists' lengths."""
    cells, trusted, erroneous = r["bufs"]
    n = kc.kmerco_get_lists_async(bf.h, trusted, r["cap"], erroneous, r["cap"])
    kc.kmerco_get_counters(bf.h, cells, r["words"])
    kc.kmerco_sync(bf.h)
    return [cells, trusted, erroneous, *n]


def run(state: dict):
    kind = state["c"]["kind"]
    if kind == "batch":
        state["batch"].insert(state["bases"], state["offsets"])
        state["batch"].classify()
        got = [_results(f, r) for f, r in zip(state["filters"], state["out"])]
        return [g[:3] for g in got], torch.tensor([g[3:] for g in got])
    bf = state["bf"]
    if kind == "query":
        n = len(state["keys"])
        est = torch.empty(n, dtype=torch.int32, device="cuda")
        kc.kmerco_query(bf.h, state["keys"], n, est)
        return est
    bf.reset()
    if kind == "merge":
        for shard in state["shards"]:
            bf.merge(shard)
    elif kind == "stream":
        for bases, offsets in state["parts"]:
            bf.insert(bases, offsets)
    else:
        bf.insert(state["bases"], state["offsets"])
    bf.classify()
    if kind != "job":
        return _results(bf, state["out"])
    s = bf.stats()
    totals = [s[k] for k in ("windows", "n_skipped", "inserted", "distinct", "trustworthy",
                             "erroneous", "saturated_counters")]
    return totals, _results(bf, state["out"])


# -------------------------------------------------------------------- work
def _distinct(c: dict, windows: int) -> int:
    """Distinct K-mers to expect: the genome's, as far as the reads cover it,
    and about one for each window that holds an error."""
    clean = (1 - c["sub"]) ** c["K"]
    genome = min(c["genome"], 4 ** c["K"] / 2)
    bad = windows * (1 - clean)
    return max(1, int(min(windows, genome * (1 - math.exp(-windows * clean / genome)) + bad,
                          4 ** c["K"])))


def _count_bytes(c: dict, reads: int, m_cells: float, distinct: int) -> float:
    key = 8 if c["K"] <= 32 else 16
    return reads * ((c["len_lo"] + c["len_hi"]) / 2 + 8) + 8 * m_cells + distinct * key


def work(case: dict) -> dict:
    """Each base and offset read once, each countBF cell and listed key written once."""
    c = case
    mean = max(1, (c["len_lo"] + c["len_hi"]) // 2 - c["K"] + 1)
    w = _windows(c)
    eta = 64 // c["alpha"]
    key = 8 if c["K"] <= 32 else 16
    if c["eq1"]:
        x, y = kc.kmerco_paper_dims(max(1, w // 2), 0.001)
        cells = x * y
    else:
        cells = (c["m"] + eta - 1) // eta
    if c["kind"] == "batch":
        b = sum(_count_bytes(c, n, d * 8 / c["alpha"] / eta, d)
                for n in _sample_sizes(c) for d in [_distinct(c, n * mean)])
    elif c["kind"] == "query":   # one counter's cell and one estimate for each key
        b = c["keys"] * (key + 8 * c["nhash"] + 4)
    elif c["kind"] == "merge":   # both shards' cells and keys in, the merged ones out
        b = 3 * 8 * cells + key * (2 * _distinct(c, w // 2) + _distinct(c, w))
    else:
        b = _count_bytes(c, c["reads"], cells, _distinct(c, w))
    return {"bytes": float(b), "flops": 0.0}


def exact(case: dict, seed: int):
    """All outputs are whole numbers and have to be equal: nothing is off by a rounding."""
    return None

"""Insertion by key ranges, its list of distinct keys and its updates, bit-exact.

Large enough calls go by key ranges (splitters, one or two levels of ranges,
shared-memory dedup, weighted increments), a further call of an ordered handle
is merged into its list.  The sizes are the edges of those steps: a chunk, a
dedup block's stage, the step from one to two levels, ranges of one key held by
very many windows, ranges of more distinct keys than the table takes, lists that
repeat each other wholly, partly or not at all.
"""
import numpy as np
import pytest

import oracle
import readsim

torch = pytest.importorskip("torch")
import paper_2305_07545_gb300 as kc  # noqa: E402
from test_gpu_parity import _dev, check, gpu_run  # noqa: E402

pytestmark = pytest.mark.gpu


def _uniform(n_reads, length, seed):
    return readsim.random_reads(n_reads, length, length, seed=seed)


@pytest.mark.parametrize("K", [5, 12, 21, 32, 33, 55, 64])
@pytest.mark.parametrize("n_reads,length", [(137, 200), (1, 33000), (40, 4096 + 70)])
def test_one_level_of_ranges(K, n_reads, length):
    b, o = _uniform(n_reads, length, seed=1000 + K + n_reads)
    g = gpu_run(b, o, K, 1 << 18, 4, 3, 2)
    check(g, b, o, K, 4, 3, 2)


@pytest.mark.parametrize("K", [21, 31, 55])
def test_two_levels_of_ranges(K):
    # 2.4e6 windows, low-complexity and uniform reads together: skewed ranges
    b1, o1 = _uniform(9000, 150, seed=K)
    b2, o2 = readsim.random_reads(9000, 100, 200, seed=K + 1, alphabet=b"ACGTN",
                                  weights=[70, 10, 10, 10, 0.1])
    b, o = np.concatenate([b1, b2]), np.concatenate([o1, o2[1:] + o1[-1]])
    g = gpu_run(b, o, K, 1 << 24, 4, 4, 2)
    check(g, b, o, K, 4, 4, 2, cross_check=False)


@pytest.mark.parametrize("K", [21, 40])
@pytest.mark.parametrize("alpha,m", [(4, 1 << 16), (8, 1 << 22), (12, 5 << 20), (5, 12 << 20),
                                     (16, 1 << 20), (2, 1 << 26)])
def test_hot_keys_and_weights(K, alpha, m):
    # two reads repeated 30,000 and 400 times among random ones: a few keys hold
    # most windows, and their increments pass the largest weight of a code
    hot = ["ACGTTGCATTGACCAGTAGGACCATTAGCAGGATTACAGATTACCAGGATT"] * 30000 + ["A" * 60] * 400
    b1, o1 = readsim.from_strings(hot)
    b2, o2 = _uniform(1500, 120, seed=alpha)
    b, o = np.concatenate([b1, b2]), np.concatenate([o1, o2[1:] + o1[-1]])
    for nhash in (3, 6):
        g = gpu_run(b, o, K, m, alpha, nhash, 2)
        check(g, b, o, K, alpha, nhash, 2, cross_check=False)


@pytest.mark.parametrize("K", [32, 31, 48])
def test_many_keys_in_one_range(K):
    # 30,000 keys with one prefix of 24 bases, one window each: the splitters that
    # fall among them still leave more keys together than a table takes, and the
    # even cut of a range sees them crowded
    st = readsim.Stream(K)
    n = 30000
    tails = readsim.ASCII[st.integers(n * (K - 16), 4).astype(np.uint8)].reshape(n, K - 16)
    heads = np.full((n, 16), ord("A"), np.uint8)
    heads[:, 15] = ord("C")
    b = np.concatenate([heads, tails], axis=1).reshape(-1)
    o = np.arange(n + 1, dtype=np.uint64) * np.uint64(K)
    b2, o2 = _uniform(60, 150, seed=K)
    b, o = np.concatenate([b, b2]), np.concatenate([o, o2[1:] + o[-1]])
    g = gpu_run(b, o, K, 1 << 20, 4, 4, 2, forward_only=True)
    check(g, b, o, K, 4, 4, 2, forward_only=True)


@pytest.mark.parametrize("K", [25, 55])
def test_calls_merged_into_an_ordered_list(K):
    # ever more of the same reads, none of them, some of them; then a call too
    # small for the ranges (the distinct set takes over) and a large one again
    b, o = readsim.scaled("tiny", 6000, seed_offset=K).generate()
    parts = []
    for c0, c1 in ((0, 2500), (0, 2500), (2500, 6000), (1000, 5500), (0, 40), (0, 6000)):
        parts.append((b[int(o[c0]):int(o[c1])].copy(), (o[c0:c1 + 1] - o[c0]).copy()))
    bases = np.concatenate([p[0] for p in parts])
    offs = [np.zeros(1, np.uint64)]
    for p in parts:
        offs.append(p[1][1:] + offs[-1][-1])
    offsets = np.concatenate(offs)
    for n in (2, 3, 4, 6):
        e = sum(len(p[1]) - 1 for p in parts[:n])
        g = gpu_run(None, None, K, 1 << 22, 8, 4, 3, batches=parts[:n])
        check(g, bases[:int(offsets[e])], offsets[:e + 1], K, 8, 4, 3)
    with kc.CountBF(K, 1 << 22, 8, 4, 3) as x, kc.CountBF(K, 1 << 22, 8, 4, 3) as y, \
            kc.CountBF(K, 1 << 22, 8, 4, 3) as z:
        y.insert(*map(_dev, parts[2]))
        torch.cuda.synchronize()
        z.insert(*map(_dev, parts[3]))
        torch.cuda.synchronize()
        x.merge(y)      # into an empty handle: copied
        x.merge(z)      # into an ordered list
        x.insert(*map(_dev, parts[5]))
        x.classify()
        keys, est = x.distinct()
        g = dict(stats=x.stats(), counters=x.counters(), keys=keys, est=est, trusted=x.trusted(),
                 erroneous=x.erroneous())
    use = [parts[2], parts[3], parts[5]]
    offs = [np.zeros(1, np.uint64)]
    for p in use:
        offs.append(p[1][1:] + offs[-1][-1])
    check(g, np.concatenate([p[0] for p in use]), np.concatenate(offs), K, 8, 4, 3)


def test_all_ones_key():
    # the 32-mer of T alone, forward strand: the value that marks a free slot
    b, o = readsim.random_reads(300, 90, 140, seed=8, alphabet=b"ACGT", weights=[1, 1, 1, 12])
    b1, o1 = readsim.from_strings(["T" * 70] * 20)
    b, o = np.concatenate([b, b1]), np.concatenate([o, o1[1:] + o[-1]])
    g = gpu_run(b, o, 32, 1 << 16, 4, 3, 2, forward_only=True)
    ref = check(g, b, o, 32, 4, 3, 2, forward_only=True)
    assert ref.distinct_lo[-1] == np.uint64(0xFFFFFFFFFFFFFFFF)


def test_batch_replay_after_a_handle_moved_its_list():
    # a captured batch insert writes a handle's list; inserting into the handle
    # alone merges that list into another buffer: the batch must not replay into
    # the old one
    parts = [readsim.scaled("tiny", 2500, seed_offset=60 + i).generate() for i in range(3)]
    dev = [(_dev(b), _dev(o)) for b, o in parts]
    stream = torch.cuda.Stream()
    fs = [kc.CountBF(21, 1 << 20, 4, 3, 2, stream=stream.cuda_stream) for _ in range(2)]
    with kc.Batch(fs) as batch:
        batch.schedule(1, 2)
        for turn in range(3):
            batch.insert([dev[0][0], dev[1][0]], [dev[0][1], dev[1][1]])
            if turn == 1:
                fs[0].insert(*dev[2])
            batch.classify()
            for i, f in enumerate(fs):
                b, o = parts[i]
                if turn == 1 and i == 0:
                    b = np.concatenate([b, parts[2][0]])
                    o = np.concatenate([o, parts[2][1][1:] + o[-1]])
                keys, est = f.distinct()
                g = dict(stats=f.stats(), counters=f.counters(), keys=keys, est=est,
                         trusted=f.trusted(), erroneous=f.erroneous())
                check(g, b, o, 21, 4, 3, 2)
    for f in fs:
        f.close()


def test_replaced_counters_decide_the_split():
    # keys with more than tau windows are trustworthy without a look at their
    # counters only while the counters are those of their windows
    b, o = readsim.scaled("tiny", 2000, seed_offset=77).generate()
    with kc.CountBF(21, 1 << 20, 4, 3, 2) as bf:
        bf.insert(_dev(b), _dev(o))
        cells = bf.counters()
        kc.kmerco_set_counters(bf.h, np.zeros_like(cells), len(cells))
        bf.classify()
        assert bf.stats()["trustworthy"] == 0
        kc.kmerco_set_counters(bf.h, cells, len(cells))
        bf.classify()
        keys, est = bf.distinct()
        g = dict(stats=bf.stats(), counters=bf.counters(), keys=keys, est=est,
                 trusted=bf.trusted(), erroneous=bf.erroneous())
    check(g, b, o, 21, 4, 3, 2)


@pytest.mark.parametrize("K", [21, 40])
def test_uneven_reads_and_few_windows(K):
    # runs of empty and short reads at the chunks' borders, long ones over several
    # chunks; then a call of which nearly no window counts, so that there are
    # fewer samples than ranges
    st = readsim.Stream(K)
    lens = np.concatenate([np.zeros(3000, np.int64), [33000], st.integers(9000, 8).astype(np.int64),
                           [1023, 1, 4096, 0, 0, 12001], st.integers(200, 300).astype(np.int64)])
    o = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    b = readsim.ASCII[st.integers(int(o[-1]), 4).astype(np.uint8)]
    g = gpu_run(b, o, K, 1 << 18, 4, 3, 2)
    check(g, b, o, K, 4, 3, 2)
    b = np.full(70000, ord("N"), np.uint8)
    o = np.array([0, 70000], np.uint64)
    for at in (0, 35000, 70000 - K - 9):
        b[at:at + K + 9] = readsim.ASCII[st.integers(K + 9, 4).astype(np.uint8)]
    g = gpu_run(b, o, K, 1 << 18, 4, 3, 2)
    check(g, b, o, K, 4, 3, 2)


@pytest.mark.parametrize("own_stream", [True, False])
@pytest.mark.parametrize("pass_codes", [0, 40000])
def test_pieces_copied_while_earlier_ones_are_counted(own_stream, pass_codes):
    # pieces of many sizes from one pinned buffer each, without a wait between them;
    # on a caller's stream a piece is written by a copy queued there right before
    parts = [readsim.scaled("tiny", n, seed_offset=300 + i).generate()
             for i, n in enumerate((3000, 40, 2500, 1, 3600, 700))]
    stream = torch.cuda.Stream()
    bf = kc.CountBF(21, 1 << 20, 4, 3, 2, pass_codes=pass_codes,
                    stream=None if own_stream else stream.cuda_stream)
    pinned = [(torch.from_numpy(b).pin_memory(), torch.from_numpy(o.view(np.int64)).pin_memory())
              for b, o in parts]
    if own_stream:
        for b, o in pinned:
            bf.insert(b, o)
    else:
        for b, o in pinned:
            src = b.cuda()
            b.zero_()
            torch.cuda.synchronize()
            with torch.cuda.stream(stream):
                torch.cuda._sleep(2_000_000)
                b.copy_(src, non_blocking=True)
            bf.insert(b, o)
            torch.cuda.synchronize()
    bf.classify()
    keys, est = bf.distinct()
    g = dict(stats=bf.stats(), counters=bf.counters(), keys=keys, est=est,
             trusted=bf.trusted(), erroneous=bf.erroneous())
    bf.close()
    offs = [np.zeros(1, np.uint64)]
    for _, o in parts:
        offs.append(o[1:] + offs[-1][-1])
    check(g, np.concatenate([b for b, _ in parts]), np.concatenate(offs), 21, 4, 3, 2)


@pytest.mark.parametrize("K", [21, 40])
@pytest.mark.parametrize("nhash", [3, 6, 7])
@pytest.mark.parametrize("alpha,m,dims", [(8, 0, (401, 409)), (4, 1 << 22, None), (8, 1100003, None)])
def test_codes_of_three_hashes(K, nhash, alpha, m, dims):
    # the partitioned increments with two and with three hashes a pass, keys that
    # are no multiple of a block's
    b, o = _uniform(1801, 151, seed=nhash + K)
    g = gpu_run(b, o, K, m, alpha, nhash, 2, dims=dims)
    check(g, b, o, K, alpha, nhash, 2, cross_check=False)


@pytest.mark.parametrize("K", [21, 40])
@pytest.mark.parametrize("passes", [2, 3, 4])
def test_passes_merged_into_the_list(K, passes):
    # a call of several passes into an empty handle, and one into a handle that holds
    # keys: every pass's keys are merged into the ascending list
    parts = [readsim.scaled("single", n, seed_offset=400 + i).generate()
             for i, n in enumerate((2400, 2000))]
    windows = 2400 * (150 - K + 1)
    dev = [(_dev(b), _dev(o)) for b, o in parts]   # read by every pass: kept until the end
    with kc.CountBF(K, 1 << 20, 4, 3, 2, pass_codes=windows * 3 // passes + 3) as bf:
        for b, o in dev:
            bf.insert(b, o)
        bf.classify()
        keys, est = bf.distinct()
        g = dict(stats=bf.stats(), counters=bf.counters(), keys=keys, est=est,
                 trusted=bf.trusted(), erroneous=bf.erroneous())
    offs = np.concatenate([parts[0][1], parts[1][1][1:] + parts[0][1][-1]])
    check(g, np.concatenate([b for b, _ in parts]), offs, K, 4, 3, 2)

"""Samples that arrive in large pieces: the keys of each are kept in order, several
pieces' together, before they are merged into the handle's list.

Every way to read or extend the list in between has to see all keys held.  What one
call makes of all pieces (checked against the oracle elsewhere) is what any sequence of
calls has to make.
"""
import numpy as np
import pytest

import readsim

torch = pytest.importorskip("torch")
import paper_2305_07545_gb300 as kc  # noqa: E402

pytestmark = pytest.mark.gpu

READS = 76000   # with 112 windows each: more than 2^23


def _pieces(n, K, seed, reads=READS):
    """n pieces on the device, overlapping in part; the last ones repeat the first."""
    st = readsim.Stream(seed)
    length = 111 + K
    genome = st.integers(80 * reads, 4).astype(np.uint8)
    out = []
    for i in range(n):
        at = st.integers(reads, len(genome) - length)
        x = genome[at[:, None] + np.arange(length)]
        if i % 2:   # half of the pieces are mostly of their own
            x = np.where(st.uniform(x.size).reshape(x.shape) < 0.02, 3 - x, x)
        b = torch.from_numpy(readsim.ASCII[x].reshape(-1)).cuda()
        o = torch.arange(reads + 1, device="cuda", dtype=torch.int64) * length
        out.append((b, o))
    torch.cuda.synchronize()
    return out + out[:2]


def _join(parts):
    offs, at = [torch.zeros(1, dtype=torch.int64, device="cuda")], 0
    for b, o in parts:
        offs.append(o[1:] + at)
        at += len(b)
    joined = torch.cat([b for b, _ in parts]), torch.cat(offs)
    torch.cuda.synchronize()
    return joined


def _state(bf):
    bf.classify()
    s = bf.stats()
    keys, est = bf.distinct()
    return [s[k] for k in ("windows", "inserted", "distinct", "trustworthy", "erroneous",
                           "saturated_counters")], [keys, est, bf.trusted(), bf.erroneous(),
                                                    bf.counters()]


def _same(got, want):
    assert got[0] == want[0]
    for g, w in zip(got[1], want[1]):
        assert np.array_equal(g, w)


def _at_once(parts, K, m):
    with kc.CountBF(K, m, 8, 3, 2) as bf:
        bf.insert(*_join(parts))
        return _state(bf)


# all merged, some pending meanwhile; the second (of two-word keys some more) merged, the
# others beside them in a set of their own; small ones, into a set built from the list
@pytest.mark.parametrize("reads", [READS, 12000, 4000, 900])
@pytest.mark.parametrize("K,m", [(31, 1 << 25), (39, 1 << 22)])
@pytest.mark.parametrize("host", [False, True])   # whether the counts held are known
def test_pieces(K, m, host, reads):
    parts = _pieces(6, K, seed=K, reads=reads)
    want = _at_once(parts, K, m)
    if host:
        parts = [(b.cpu().pin_memory(), o.cpu().pin_memory()) for b, o in parts]
    with kc.CountBF(K, m, 8, 3, 2) as bf:
        for _ in range(2):   # again after a reset
            for b, o in parts:
                bf.insert(b, o)
            _same(_state(bf), want)
            bf.reset()
        for b, o in parts[:4]:   # keys pending at a reset are gone
            bf.insert(b, o)
        bf.reset()
        for b, o in parts:
            bf.insert(b, o)
        _same(_state(bf), want)


@pytest.mark.parametrize("reads", [READS, 4000])
@pytest.mark.parametrize("K", [31, 39])
def test_calls_between_pieces(K, reads):
    m = 1 << 22
    parts = _pieces(5, K, seed=K + 1, reads=reads)
    small = parts[0][0][:(111 + K) * 90].clone(), parts[0][1][:91].clone()
    torch.cuda.synchronize()
    with kc.CountBF(K, m, 8, 3, 2) as bf:
        for n, (b, o) in enumerate(parts, 1):
            bf.insert(b, o)
            if n in (4, 6):   # the totals of the keys held, some of them pending
                assert bf.stats()["distinct"] == _at_once(parts[:n], K, m)[0][2]
            if n == 5:
                _same(_state(bf), _at_once(parts[:n], K, m))
        bf.insert(*small)     # to the set
        _same(_state(bf), _at_once(parts + [small], K, m))
    with kc.CountBF(K, m, 8, 3, 2) as bf:
        for b, o in parts[:3]:
            bf.insert(b, o)
        kw = 2 if K > 32 else 1
        extra = np.arange(1000 * kw, dtype=np.uint64) * np.uint64(3)   # host keys, staged
        kc.kmerco_add_distinct(bf.h, extra, 1000)
        bf.classify()
        got = bf.distinct()[0].reshape(-1, kw)
    keys = np.concatenate([_at_once(parts[:3], K, m)[1][0].reshape(-1, kw), extra.reshape(-1, kw)])
    order = np.lexsort(keys.T)
    keys = keys[order]
    new = np.concatenate([[True], (keys[1:] != keys[:-1]).any(axis=1)])
    assert np.array_equal(got, keys[new])


@pytest.mark.parametrize("reads", [READS, 4000])
def test_handles_with_keys_pending_are_merged(reads):
    K, m = 31, 1 << 22
    parts = _pieces(5, K, seed=7, reads=reads)
    for cut in (3, 4):
        with kc.CountBF(K, m, 8, 3, 2) as x, kc.CountBF(K, m, 8, 3, 2) as y:
            for b, o in parts[:cut]:
                x.insert(b, o)
            for b, o in parts[cut:]:
                y.insert(b, o)
            x.merge(y)
            _same(_state(x), _at_once(parts, K, m))
            _same(_state(y), _at_once(parts[cut:], K, m))


@pytest.mark.parametrize("reads", [READS, 4000])
@pytest.mark.parametrize("schedule", [0, 1])
def test_a_batch_with_keys_pending(schedule, reads):
    K, m = 31, 1 << 22
    parts = _pieces(4, K, seed=8, reads=reads)
    stream = torch.cuda.Stream()
    fs = [kc.CountBF(K, m, 8, 3, 2, stream=stream.cuda_stream) for _ in range(2)]
    with kc.Batch(fs) as batch:
        batch.schedule(schedule, 2)
        batch.insert([parts[0][0], parts[1][0]], [parts[0][1], parts[1][1]])
        for b, o in parts[2:4]:   # into one handle alone: with the schedule by samples its
            fs[0].insert(b, o)    # list is in order and keys are pending
        batch.classify()
        _same(_state(fs[0]), _at_once([parts[0]] + parts[2:4], K, m))
        for b, o in parts[2:4]:
            fs[0].insert(b, o)
        batch.insert([parts[1][0], parts[2][0]], [parts[1][1], parts[2][1]], reset=False)
        batch.classify()
        _same(_state(fs[0]), _at_once([parts[0]] + parts[2:4] * 2 + [parts[1]], K, m))
        _same(_state(fs[1]), _at_once([parts[1], parts[2]], K, m))
        fs[0].insert(*parts[3])
        fs[0].insert(*parts[2])
        batch.insert([parts[0][0], parts[1][0]], [parts[0][1], parts[1][1]])   # resets
        batch.classify()
        _same(_state(fs[0]), _at_once([parts[0]], K, m))
    for f in fs:
        f.close()


def test_pieces_under_a_budget():
    # what the list and the set of all pieces need is enough, pending keys or not
    K, m = 31, 1 << 22
    parts = _pieces(5, K, seed=9)
    want = _at_once(parts, K, m)
    with kc.CountBF(K, m, 8, 3, 2, hbm_budget=1 << 40) as bf:
        for b, o in parts:
            bf.insert(b, o)
        bf.classify()
        most = bf.stats()["device_bytes"]
    windows = READS * 112
    refused = 0
    for share in (0.95, 0.8, 0.65, 0.55):
        with kc.CountBF(K, m, 8, 3, 2, hbm_budget=int(share * most)) as bf:
            try:
                for b, o in parts:
                    bf.insert(b, o)
                bf.classify()
            except kc.KmercoError as e:
                assert e.status == kc.ENOMEM
                # never under the list and the set with their growth, and classification
                assert share * most < 64 * (want[0][2] + windows) + 60 * want[0][2]
                refused += 1
                continue
            _same(_state(bf), want)
    assert refused < 4


@pytest.mark.parametrize("K", [31, 39])
def test_a_refused_piece_leaves_the_list_where_it_was(K):
    # a large third piece finds no room, first by ranges, then for the set of its own
    # beside the list set aside: the results of the first two are there as before
    m, kw = 1 << 22, 1 if K <= 32 else 2
    parts = _pieces(2, K, seed=K, reads=4000)[:2]
    large = _pieces(1, K, seed=K + 5, reads=60000)[0]
    with kc.CountBF(K, m, 8, 3, 2) as bf:
        for b, o in parts:
            bf.insert(b, o)
        bf.classify()
        bf.distinct()
        held = bf.stats()["device_bytes"]
    # the large piece's list and set alone take 160 MB a key word, twice what is held
    assert 24 * 60000 * 112 * kw > 2 * held
    with kc.CountBF(K, m, 8, 3, 2, hbm_budget=held + (4 << 20)) as bf:
        for b, o in parts:
            bf.insert(b, o)
        want = _state(bf)
        with pytest.raises(kc.KmercoError) as e:
            bf.insert(*large)
        assert e.value.status == kc.ENOMEM
        filler = [torch.full((n,), -1, dtype=torch.int64, device="cuda") for n in (1 << 16, 1 << 20)]
        torch.cuda.synchronize()
        _same(_state(bf), want)
        del filler


@pytest.mark.parametrize("K", [31, 39])
def test_a_call_of_several_passes_beside_pending_keys(K):
    # the third piece's keys are pending; the fourth call is all pieces once more, in three
    # passes, each merged into the list, which takes turns between its two places
    m = 1 << 22
    parts = _pieces(2, K, seed=K + 9)
    whole = _join(parts)
    with kc.CountBF(K, m, 8, 3, 2, pass_codes=3 * READS * 112 * 4 // 3) as bf:
        for b, o in parts[:3]:
            bf.insert(b, o)
        bf.insert(*whole)
        _same(_state(bf), _at_once(parts[:3] + [whole], K, m))


def test_pieces_without_a_window_that_counts():
    # pending keys whose count is none: pieces of N between others, all sizes known late
    K, m = 31, 1 << 22
    parts = _pieces(3, K, seed=12)
    empty = [(torch.full_like(b, ord("N")), o) for b, o in parts[:2]]
    torch.cuda.synchronize()
    order = [parts[0], parts[1], empty[0], parts[2], empty[1], empty[0], parts[1], parts[2]]
    want = _at_once(order, K, m)
    for host in (False, True):
        use = [(b.cpu().pin_memory(), o.cpu().pin_memory()) for b, o in order] if host else order
        with kc.CountBF(K, m, 8, 3, 2) as bf:
            for b, o in use:
                bf.insert(b, o)
            _same(_state(bf), want)

"""Where the key space is cut into ranges, bit-exact and in its cost.

Long keys with a common beginning (a constant flank, a primer, an adapter) have
equal 64-bit prefixes and are cut by their low words; ranges that the samples
say nothing about hold far more keys than a block's table and are counted in
rounds.  Keys leave the ranges in key order, or in none: so do the later passes of
a call into a list with a cap, whose keys go to the distinct set.
"""
import numpy as np
import pytest

import readsim

torch = pytest.importorskip("torch")
import paper_2305_07545_gb300 as kc  # noqa: E402
from test_gpu_parity import _dev, check  # noqa: E402
from test_gpu_set_keys import _count, _join  # noqa: E402

pytestmark = pytest.mark.gpu


def _bases(st, *shape):
    return readsim.ASCII[st.integers(int(np.prod(shape)), 4).astype(np.uint8)].reshape(shape)


def _even(x):
    return x.reshape(-1), np.arange(len(x) + 1, dtype=np.uint64) * np.uint64(x.shape[1])


def _flanked(n, length, flank, seed):
    st = readsim.Stream(seed)
    head = np.broadcast_to(_bases(st, 1, flank), (n, flank))
    return _even(np.concatenate([head, _bases(st, n, length - flank)], axis=1))


@pytest.mark.parametrize("K,length,flank", [(33, 70, 40), (55, 70, 40), (64, 90, 50)])
@pytest.mark.parametrize("n", [9000, 60000])   # one level of ranges, and two
@pytest.mark.parametrize("forward_only", [False, True])
def test_keys_with_a_common_beginning(K, length, flank, n, forward_only):
    parts = [_flanked(n, length, flank, seed=K + n)]
    g = _count(parts, K, 1 << 22, 8, 3, 2, forward_only=forward_only)
    check(g, *_join(parts), K, 8, 3, 2, forward_only=forward_only, cross_check=False)


def _unordered(windows, passes):
    """Options that make the passes after a call's first one unordered (three hashes)."""
    return dict(max_distinct=1 << 28, pass_codes=3 * (windows // passes + 1))


@pytest.mark.parametrize("K", [40, 55])
@pytest.mark.parametrize("second", ["call", "passes"])   # merged into the list, put in the set
def test_a_further_part_with_a_common_beginning(K, second):
    parts = [readsim.random_reads(3000, 150, 150, seed=K), _flanked(9000, 72, 40, seed=K + 1),
             _flanked(9000, 72, 40, seed=K + 1)]
    b, o = _join(parts)
    if second == "call":
        g = _count(parts, K, 1 << 22, 8, 3, 2)
    else:
        windows = 3000 * (151 - K) + 18000 * (73 - K)
        g = _count([(b, o)], K, 1 << 22, 8, 3, 2, **_unordered(windows, 4))
    check(g, b, o, K, 8, 3, 2, cross_check=False)


@pytest.mark.parametrize("K,forward_only", [(21, False), (32, True), (33, False), (55, False),
                                            (64, True)])
@pytest.mark.parametrize("unordered", [False, True])
def test_ranges_that_the_samples_miss(K, forward_only, unordered):
    # 25,000 windows among 6e7 bases of reads too short to hold one: the samples,
    # spread over the bases, meet next to none of them, so a range has thousands of keys
    st = readsim.Stream(K)
    some = _bases(st, 250, K + 99)
    some[0] = ord("T")   # forward strand: the largest key there is
    short = _bases(st, 3_000_000, 20)
    cut = 3 * len(short) // 4   # in the second of two passes
    b, o = _join([_even(short[:cut]), _even(some), _even(short[cut:])])
    kw = _unordered(25000, 2) if unordered else {}
    g = _count([(b, o)], K, 1 << 22, 8, 3, 2, forward_only=forward_only, **kw)
    check(g, b, o, K, 8, 3, 2, forward_only=forward_only, cross_check=False)


def _insert_ms(b, o, K, m=1 << 24):
    d = _dev(b), _dev(o)
    with kc.CountBF(K, m, 4, 4, 3) as bf:
        ms = []
        for _ in range(4):
            bf.reset()
            bf.insert(*d)
            bf.classify()
            ms.append(bf.stats()["insert_ms"])
    return min(ms)


def test_a_common_beginning_costs_no_rounds():
    # as many windows and distinct keys as random reads have; cut by prefixes alone a
    # block took a hundred times as long for its share of the keys.  Eight times
    # leaves room for more bisecting and crowded cuts.
    n, K = 60000, 55
    flanked = _insert_ms(*_flanked(n, 70, 40, seed=1), K)
    uniform = _insert_ms(*readsim.random_reads(n, 70, 70, seed=2), K)
    assert flanked < 8 * uniform, (flanked, uniform)


@pytest.mark.parametrize("K,forward_only", [(13, False), (21, False), (32, True), (33, True),
                                            (55, False), (64, True)])
@pytest.mark.parametrize("n", [1500, 12000])   # one level of ranges, and two
def test_keys_held_by_very_many_windows(K, forward_only, n):
    # reads of one base each (the smallest and the largest keys there are), of T's and a
    # last A (the largest key but three), one read and one with another last base many times
    st = readsim.Stream(n + K)
    x = _bases(st, n, 150)
    x[: n // 8] = ord("T")
    x[n // 8: n // 6] = ord("A")
    x[n // 6: n // 4, :K] = ord("T")
    x[n // 6: n // 4, K - 1] = ord("A")
    x[n // 4: n // 3] = x[n // 4]
    x[n // 3: n // 2] = x[n // 4]
    x[n // 3: n // 2, K - 1] = ord("C")
    parts = [_even(x[_shuffled(n, st)])]
    g = _count(parts, K, 1 << 22, 8, 3, 2, forward_only=forward_only)
    check(g, *_join(parts), K, 8, 3, 2, forward_only=forward_only, cross_check=False)
    g = _count(parts, K, 1 << 22, 8, 3, 2, forward_only=forward_only,
               **_unordered(n * (151 - K), 3))
    check(g, *_join(parts), K, 8, 3, 2, forward_only=forward_only, cross_check=False)


def _shuffled(n, st):
    return np.argsort(st.uniform(n))


@pytest.mark.parametrize("K", [31, 55])
def test_a_key_of_very_many_windows_costs_no_more_than_others(K):
    # a tenth of the reads of one base: their windows were one block's, which took 15
    # times as long as all the others for the rest
    n = 200000
    b, o = readsim.random_reads(n, 150, 150, seed=1)
    uniform = _insert_ms(b, o, K, m=1 << 26)
    x = b.reshape(n, 150).copy()
    x[::10] = ord("G")
    hot = _insert_ms(x.reshape(-1), o, K, m=1 << 26)
    assert hot < 2 * uniform, (hot, uniform)

"""Keys that look like a free slot of the distinct set, bit-exact.

With 32 and 64 bases a key takes whole words, so a free slot is marked by all
ones: the value of the K-mer of T alone, read forward (or where the hash picks
the strand).
"""
import numpy as np
import pytest

import readsim

torch = pytest.importorskip("torch")
import paper_2305_07545_gb300 as kc  # noqa: E402
from test_gpu_parity import _dev, check  # noqa: E402

pytestmark = pytest.mark.gpu


def _join(parts):
    offs = [np.zeros(1, np.uint64)]
    for _, o in parts:
        offs.append(o[1:] + offs[-1][-1])
    return np.concatenate([b for b, _ in parts]), np.concatenate(offs)


def _count(parts, K, m, alpha, nhash, tau, **kw):
    dev = [(_dev(b), _dev(o)) for b, o in parts]
    with kc.CountBF(K, m, alpha, nhash, tau, **kw) as bf:
        for b, o in dev:
            bf.insert(b, o)
        bf.classify()
        keys, est = bf.distinct()
        return dict(stats=bf.stats(), counters=bf.counters(), keys=keys, est=est,
                    trusted=bf.trusted(), erroneous=bf.erroneous())


def _poly_t(n, seed):
    """n random reads, one of T's among them."""
    b, o = readsim.random_reads(n, 80, 150, seed=seed)
    b1, o1 = readsim.from_strings(["T" * 100])
    return _join([(b, o), (b1, o1)])


@pytest.mark.parametrize("K", [32, 64])
@pytest.mark.parametrize("mode", [dict(forward_only=True), dict(canonical_hash=True)])
# calls that go to the set: small ones; a list in order and a small one; a large list
# and one of a tenth of it
@pytest.mark.parametrize("sizes", [(20, 20), (400, 20), (14000, 1800, 20)])
def test_the_key_of_all_ones(K, mode, sizes):
    parts = [_poly_t(n, seed=K + i) for i, n in enumerate(sizes)]
    g = _count(parts, K, 1 << 20, 8, 3, 2, **mode)
    ref = check(g, *_join(parts), K, 8, 3, 2, cross_check=False, **mode)
    if "forward_only" in mode:
        assert ref.distinct_lo[-1] == np.uint64(0xFFFFFFFFFFFFFFFF)


@pytest.mark.parametrize("K", [32, 64])
def test_the_key_of_all_ones_added_merged_and_after_a_reset(K):
    b, o = _poly_t(30, seed=3)
    ones = np.full(K // 32, 2 ** 64 - 1, np.uint64)
    d = _dev(b), _dev(o)
    with kc.CountBF(K, 1 << 18, 4, 3, 2, forward_only=True) as bf, \
            kc.CountBF(K, 1 << 18, 4, 3, 2, forward_only=True) as other:
        for _ in range(2):   # the place is free again after a reset
            kc.kmerco_add_distinct(bf.h, ones, 1)
            kc.kmerco_add_distinct(bf.h, ones, 1)
            assert bf.stats()["distinct"] == 1
            bf.insert(*d)
            bf.classify()
            keys, est = bf.distinct()
            g = dict(stats=bf.stats(), counters=bf.counters(), keys=keys, est=est,
                     trusted=bf.trusted(), erroneous=bf.erroneous())
            check(g, b, o, K, 4, 3, 2, forward_only=True)
            n = len(keys)
            other.reset()
            kc.kmerco_add_distinct(other.h, ones, 1)
            other.merge(bf)
            other.classify()
            assert other.stats()["distinct"] == n
            bf.reset()


@pytest.mark.parametrize("sizes", [(1, 1), (40, 40, 40)])
def test_64_mers_with_a_half_of_t(sizes):
    # one word of such a key is all ones, as both are of a free slot; every key comes
    # several times, and other keys probe past it
    st = readsim.Stream(64)
    half = readsim.ASCII[st.integers(60 * 32, 4).astype(np.uint8)].reshape(60, 32)
    t = np.full((60, 32), ord("T"), np.uint8)
    some = np.concatenate([np.concatenate([half, t], axis=1), np.concatenate([t, half], axis=1)])
    own = some.reshape(-1), np.arange(121, dtype=np.uint64) * np.uint64(64)
    parts = [_join([own, readsim.random_reads(n, 64, 100, seed=n + i), own])
             for i, n in enumerate(sizes)]
    g = _count(parts, 64, 1 << 14, 8, 3, 2, forward_only=True)
    check(g, *_join(parts), 64, 8, 3, 2, forward_only=True)
    more = _count(parts, 64, 1 << 14, 8, 3, 2)
    check(more, *_join(parts), 64, 8, 3, 2)

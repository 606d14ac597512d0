"""The sorts of a distinct list that is in no order, against numpy.

An insert by key ranges leaves an ordered list, so keys are handed in here
(kmerco_add_distinct), each shape at the size that takes it to the sort that its
edges are in: buckets of a block's shared memory with a bin too large for one, with
keys crowded in few of a bucket's cells, with more buckets than the scatter counts;
and segments under equal top bits too long for a block.
"""
import numpy as np
import pytest

import readsim

torch = pytest.importorskip("torch")
import paper_2305_07545_gb300 as kc  # noqa: E402
from test_gpu_parity import check  # noqa: E402
from test_gpu_set_keys import _count  # noqa: E402

pytestmark = pytest.mark.gpu


def _raw(n, bits, seed):
    return readsim.Stream(seed).raw(n) >> np.uint64(64 - bits)


def _sorted_list(keys, K):
    n = len(keys)
    with kc.CountBF(K, 1 << 12, 4, 2, 1) as bf:
        kc.kmerco_add_distinct(bf.h, np.ascontiguousarray(keys).reshape(-1), n)
        kc.kmerco_add_distinct(bf.h, np.ascontiguousarray(keys[::-7]).reshape(-1), len(keys[::-7]))
        bf.classify()
        return bf.distinct()[0]


ONE_WORD = {
    # 1.2e6 keys, 30,000 of them under one histogram bin: more than a block sorts
    "large bin": lambda: np.concatenate([_raw(1_200_000, 62, 1), _raw(30_000, 40, 2)]),
    # a third of the keys in two places of their buckets' ranges
    "crowded cells": lambda: np.concatenate(
        [_raw(900_000, 62, 3), (np.uint64(1) << np.uint64(61)) + _raw(2_000, 12, 4),
         (_raw(300_000, 10, 5) << np.uint64(52)) + _raw(300_000, 9, 6)]),
}


@pytest.mark.parametrize("shape", sorted(ONE_WORD))
def test_one_word_lists(shape):
    keys = ONE_WORD[shape]()
    assert np.array_equal(_sorted_list(keys, 31), np.unique(keys))


def _many_buckets():
    # bins of just over half a bucket: 25,000 of them cannot be merged two by two
    bins = torch.arange(25_000, device="cuda").repeat_interleave(4100)
    return (bins << 46) + (torch.arange(4100, device="cuda") << 3).repeat(25_000)


def _segments():
    # above the bucket sort's range: segments under the top 24 bits, runs of them too
    # long for a block, and one for a block's own sort
    g = torch.Generator(device="cuda").manual_seed(8)
    return torch.cat([torch.randint(1 << 62, (134_300_000,), generator=g, device="cuda"),
                      torch.randint(1 << 37, (70_000,), generator=g, device="cuda"),
                      (5 << 50) + torch.randint(1 << 38, (9_000,), generator=g, device="cuda")])


@pytest.mark.parametrize("shape", [_many_buckets, _segments])
def test_large_one_word_lists(shape):
    keys = shape()
    keys = keys[torch.randperm(len(keys), device="cuda")]
    want = torch.unique(keys)
    torch.cuda.synchronize()
    with kc.CountBF(31, 1 << 12, 4, 2, 1) as bf:
        kc.kmerco_add_distinct(bf.h, keys, len(keys))
        bf.classify()
        n = bf.stats()["distinct"]
        got = torch.empty(n, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        assert kc.kmerco_get_distinct(bf.h, got, None, n) == n
    assert torch.equal(got, want)


@pytest.mark.parametrize("n", [300_000, 2_200_000])   # radix sort, segments
def test_two_word_lists(n):
    K = 45
    lo, hi = readsim.Stream(n).raw(n), _raw(n, 26, n + 1)
    hi[: n // 8] = 12345                      # runs under equal top bits
    lo[: n // 50] &= np.uint64(0xFFFF)        # of few different low words
    got = _sorted_list(np.stack([lo, hi], axis=1), K)
    order = np.lexsort((lo, hi))
    lo, hi = lo[order], hi[order]
    new = np.concatenate([[True], (lo[1:] != lo[:-1]) | (hi[1:] != hi[:-1])])
    assert np.array_equal(got[:, 0], lo[new]) and np.array_equal(got[:, 1], hi[new])


@pytest.mark.parametrize("K", [21, 40])
@pytest.mark.parametrize("alpha", [4, 16])
@pytest.mark.parametrize("m", [1 << 7, 1 << 13])   # one region's buffer is passed, no slice's
def test_weighted_codes_beyond_a_region(K, alpha, m):
    # 30,000 distinct keys, a third of them many times, into a few cells: the regions in
    # use get more codes than their share, with weights above one
    b1, o1 = readsim.random_reads(200, 120, 120, seed=K)
    b2, o2 = readsim.random_reads(100, 120, 120, seed=K + 1)
    b = np.concatenate([b1] + [b2] * 40)
    o = np.arange(200 + 40 * 100 + 1, dtype=np.uint64) * np.uint64(120)
    g = _count([(b, o)], K, m, alpha, 4, 3, update_mode=kc.UPDATE_PARTITIONED)
    check(g, b, o, K, alpha, 4, 3, cross_check=False)

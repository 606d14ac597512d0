"""A call that fails for memory leaves the handle as it was.

The handle's results are read again after the refused call: keys, estimates,
both lists and the countBF have to be those of the calls that succeeded.  The
caller's allocator hands freed blocks out again at once, so results that are
read from a freed buffer would hold the filler that the test puts there.
"""
import numpy as np
import pytest

import readsim

torch = pytest.importorskip("torch")
import paper_2305_07545_gb300 as kc  # noqa: E402
from test_gpu_parity import _dev, check  # noqa: E402

pytestmark = pytest.mark.gpu


def _results(bf):
    keys, est = bf.distinct()
    return dict(stats=bf.stats(), counters=bf.counters(), keys=keys, est=est,
                trusted=bf.trusted(), erroneous=bf.erroneous())


def _held(K, b, o, **kw):
    """Device bytes of a handle after one insert and a classification."""
    with kc.CountBF(K, 1 << 18, 4, 3, 2, **kw) as bf:
        bf.insert(_dev(b), _dev(o))
        bf.classify()
        return bf.stats()["device_bytes"]


@pytest.mark.parametrize("K", [21, 40])
@pytest.mark.parametrize("allocator", [None, "torch"])
def test_results_after_an_insert_whose_set_does_not_fit(K, allocator):
    # the second call moves the list (1.1e6 bytes a key word) and then finds no room
    # for the set, which is twice as large
    b, o = readsim.random_reads(17000 // (150 - K + 1) + 1, 150, 150, seed=5)
    b2, o2 = readsim.random_reads(120000 // (150 - K + 1) + 1, 150, 150, seed=6)
    kw = 1 if K <= 32 else 2
    budget = _held(K, b, o) + 1_200_000 * kw
    with kc.CountBF(K, 1 << 18, 4, 3, 2, hbm_budget=budget, allocator=allocator) as bf:
        bf.insert(_dev(b), _dev(o))
        bf.classify()
        d2 = _dev(b2), _dev(o2)
        with pytest.raises(kc.KmercoError) as e:
            bf.insert(*d2)
        assert e.value.status == kc.ENOMEM
        filler = [torch.full((n,), -1, dtype=torch.int64, device="cuda")
                  for n in (1 << 14, 17000 * kw, 1 << 16, 1 << 18)]
        torch.cuda.synchronize()
        check(_results(bf), b, o, K, 4, 3, 2)
        probes = bf.distinct()[0][::97].copy()
        ranks = np.zeros(len(probes), np.uint64)
        kc.kmerco_rank_of(bf.h, probes, len(probes), ranks)
        assert np.array_equal(ranks, np.arange(0, bf.stats()["distinct"], 97, dtype=np.uint64))
        del filler


@pytest.mark.parametrize("K", [20, 21, 40])   # the sort ends in either of its buffers
def test_results_after_an_add_whose_set_does_not_fit(K):
    # calls of a few windows go to the distinct set, so the list is sorted into a
    # buffer of its own; the added keys are staged on the device before the set is
    # found not to fit
    parts = [readsim.random_reads(40, 150, 150, seed=7 + i) for i in range(2)]
    kw = 1 if K <= 32 else 2
    more = np.arange(60000 * kw, dtype=np.uint64)
    with kc.CountBF(K, 1 << 18, 4, 3, 2) as bf:
        for b, o in parts:
            bf.insert(_dev(b), _dev(o))
        bf.classify()
        held = bf.stats()["device_bytes"]
    # the staging (a quarter more than the keys) and the list fit, the set does not
    with kc.CountBF(K, 1 << 18, 4, 3, 2, hbm_budget=held + 1_300_000 * kw) as bf:
        for b, o in parts:
            bf.insert(_dev(b), _dev(o))
        bf.classify()
        with pytest.raises(kc.KmercoError) as e:
            kc.kmerco_add_distinct(bf.h, more, 60000)
        assert e.value.status == kc.ENOMEM
        (b1, o1), (b2, o2) = parts
        check(_results(bf), np.concatenate([b1, b2]), np.concatenate([o1, o2[1:] + o1[-1]]),
              K, 4, 3, 2)


@pytest.mark.parametrize("K", [21, 40])
@pytest.mark.parametrize("share", [24.3, 27, 30, 33, 34.5, 36, 40, 60])
def test_a_budget_that_holds_the_list_and_the_set_is_enough(K, share):
    # 24 bytes a window and key word hold the list and the set; the scratch of an
    # insert by key ranges is taken only where it leaves room for what has to be had,
    # and goes when the classification needs the memory
    reads = 60
    b, o = readsim.random_reads(reads, 150, 150, seed=11)
    b, o = np.tile(b, 30), np.arange(30 * reads + 1, dtype=np.uint64) * np.uint64(150)
    kw = 1 if K <= 32 else 2
    windows = 30 * reads * (150 - K + 1)
    with kc.CountBF(K, 1 << 18, 4, 3, 2) as bf:
        base = bf.stats()["device_bytes"]
    distinct = reads * (150 - K + 1)
    # classification: two sort buffers, the lists, bits, and the sorts' small scratch
    budget = base + int(share * kw * windows) + 60 * kw * distinct + (1 << 16)
    with kc.CountBF(K, 1 << 18, 4, 3, 2, hbm_budget=budget) as bf:
        bf.insert(_dev(b), _dev(o))
        bf.classify()
        check(_results(bf), b, o, K, 4, 3, 2)
        assert bf.stats()["device_bytes"] <= budget


def test_scratch_of_an_insert_makes_room_for_later_calls():
    # an insert by key ranges that fits holds its scratch on; classification and the
    # query's staging need more than what is left beside it
    K = 31
    b, o = readsim.random_reads(2000, 150, 150, seed=12)
    with kc.CountBF(K, 1 << 18, 4, 3, 2) as bf:
        bf.insert(_dev(b), _dev(o))
        kc.kmerco_sync(bf.h)
        budget = bf.stats()["device_bytes"] + 4096
    with kc.CountBF(K, 1 << 18, 4, 3, 2, hbm_budget=budget) as bf:
        bf.insert(_dev(b), _dev(o))
        bf.classify()
        check(_results(bf), b, o, K, 4, 3, 2)
        q = np.arange(100000, dtype=np.uint64)
        assert len(bf.query(q)) == len(q)

"""Handles with a cap on the distinct list or a bound of the retry loops, in calls
large enough for key ranges."""
import numpy as np
import pytest

import oracle
import readsim

torch = pytest.importorskip("torch")
import paper_2305_07545_gb300 as kc  # noqa: E402
from test_gpu_parity import _dev, check  # noqa: E402
from test_gpu_set_keys import _join  # noqa: E402

pytestmark = pytest.mark.gpu


def _results(bf):
    keys, est = bf.distinct()
    return dict(stats=bf.stats(), counters=bf.counters(), keys=keys, est=est,
                trusted=bf.trusted(), erroneous=bf.erroneous())


@pytest.mark.parametrize("K", [21, 40])
@pytest.mark.parametrize("m", [1 << 18, 1 << 24])   # atomic and partitioned update
@pytest.mark.parametrize("pass_codes", [0, 60000])  # one pass, and several
def test_a_cap_on_the_list(K, m, pass_codes):
    parts = [readsim.scaled("tiny", n, seed_offset=K + n).generate() for n in (1500, 700, 2500)]
    dev = [(_dev(b), _dev(o)) for b, o in parts]
    distinct = []
    for n in (1, 2, 3):
        b, o = _join(parts[:n])
        distinct.append(len(oracle.run(b, o, K, m, 4, 3, 2, cross_check=False).distinct_lo))
    # the cap is the first call's keys, then one key less than all calls', then as many
    for cap, fit in ((distinct[0], 1), (distinct[2] - 1, 2), (distinct[2], 3),
                     (distinct[0] - 1, 0)):
        with kc.CountBF(K, m, 4, 3, 2, max_distinct=cap, pass_codes=pass_codes) as bf:
            for n in (1, 2, 3):
                bf.insert(*dev[n - 1])
                b, o = _join(parts[:n])
                if n <= fit:
                    bf.classify()
                    check(_results(bf), b, o, K, 4, 3, 2, cross_check=False)
                    continue
                with pytest.raises(kc.KmercoError) as e:
                    bf.classify()
                assert e.value.status == kc.ENOMEM
                # every window is counted all the same
                want = oracle.run(b, o, K, m, 4, 3, 2, cross_check=False).filter
                cells = np.empty_like(want)
                kc.kmerco_get_counters(bf.h, cells, len(cells))
                assert np.array_equal(cells, want)
            bf.reset()
            bf.insert(_dev(parts[1][0][:2100]), _dev(parts[1][1][:22]))
            bf.classify()
            check(_results(bf), parts[1][0][:2100], parts[1][1][:22], K, 4, 3, 2)


@pytest.mark.parametrize("K", [21, 40])
@pytest.mark.parametrize("limit", [1023, 1024, 1 << 16])   # window by window, by key ranges
@pytest.mark.parametrize("mode", [kc.UPDATE_ATOMIC, kc.UPDATE_PARTITIONED])
def test_a_retry_limit_that_is_not_met(K, limit, mode):
    parts = [readsim.scaled("tiny", n, seed_offset=K + n).generate() for n in (1500, 2500)]
    with kc.CountBF(K, 1 << 24, 8, 4, 2, retry_limit=limit, update_mode=mode) as bf, \
            kc.CountBF(K, 1 << 24, 8, 4, 2, retry_limit=limit, update_mode=mode) as into:
        for b, o in parts:
            bf.insert(b, o)
        bf.classify()
        check(_results(bf), *_join(parts), K, 8, 4, 2, cross_check=False)
        into.merge(bf)
        into.classify()
        assert np.array_equal(into.distinct()[0], bf.distinct()[0])
        assert np.array_equal(into.counters(), bf.counters())


def test_a_retry_limit_costs_no_partitioned_update():
    # a countBF beyond L2: the window-by-window kernel takes over twice as long
    n, K = 400000, 31
    b, o = readsim.random_reads(n, 150, 150, seed=9)
    d = _dev(b), _dev(o)
    ms = []
    for kw in (dict(), dict(retry_limit=1 << 16)):
        with kc.CountBF(K, 1 << 28, 4, 4, 3, **kw) as bf:
            t = []
            for _ in range(4):
                bf.reset()
                bf.insert(*d)
                bf.classify()
                t.append(bf.stats()["insert_ms"])
            ms.append(min(t))
    assert ms[1] < 1.5 * ms[0], ms

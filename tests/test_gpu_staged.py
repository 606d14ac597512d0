"""Windows inserted one by one with their increments partitioned, bit-exact: the
insert kernel writes the keys down and updates no counter.  The sizes go around a
chunk and a pass of the increments; calls come before and after ones by key ranges,
and counters of one region or slice take more codes than its buffer holds."""
import numpy as np
import pytest

import readsim

torch = pytest.importorskip("torch")
import paper_2305_07545_gb300 as kc  # noqa: E402
from test_gpu_parity import check  # noqa: E402
from test_gpu_set_keys import _count, _join  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 21, 32, 33, 55])
@pytest.mark.parametrize("alpha,m,nhash", [(4, 1 << 16, 3), (5, 12 << 18, 4), (8, 1 << 22, 1),
                                           (16, 1 << 22, 4), (1, 1 << 20, 2)])
@pytest.mark.parametrize("pass_codes", [0, 3000])   # one pass of increments, and several
def test_small_calls_with_the_partitioned_update(K, alpha, m, nhash, pass_codes):
    tau = 0 if alpha == 1 else 2
    parts = [readsim.random_reads(n, 0, 160, seed=K + n, alphabet=b"ACGTN",
                                  weights=[25, 25, 25, 25, 0.2]) for n in (1, 37, 110)]
    g = _count(parts, K, m, alpha, nhash, tau, update_mode=kc.UPDATE_PARTITIONED,
               pass_codes=pass_codes)
    check(g, *_join(parts), K, alpha, nhash, tau)


@pytest.mark.parametrize("K", [25, 41])
@pytest.mark.parametrize("m", [1 << 20, 1 << 26])   # slices are regions; regions of many slices
def test_a_call_after_one_by_ranges(K, m):
    # 8e5 and 1.2e5 windows after a list in order, by the automatic rule: partitioned, then not
    parts = [readsim.scaled("tiny", 3000, seed_offset=K).generate(),
             readsim.scaled("single", 7000, seed_offset=K).generate(),
             readsim.scaled("tiny", 1800, seed_offset=K + 1).generate()]
    g = _count(parts, K, m, 4, 4, 3)
    check(g, *_join(parts), K, 4, 4, 3, cross_check=False)


@pytest.mark.parametrize("alpha", [4, 16])   # counting and compare-and-swap apply
@pytest.mark.parametrize("K", [21, 40])
def test_more_codes_than_a_region_holds(K, alpha):
    # 60 distinct keys in 8e5 windows: their regions and slices take twenty times their
    # share, the rest is added to the countBF directly
    b, o = readsim.random_reads(1, K + 59, K + 59, seed=K)
    n = 13000
    parts = [readsim.scaled("tiny", 3000, seed_offset=K).generate(),
             (np.tile(b, n), np.arange(n + 1, dtype=np.uint64) * np.uint64(len(b)))]
    g = _count(parts, K, 1 << 24, alpha, 4, 3, update_mode=kc.UPDATE_PARTITIONED)
    check(g, *_join(parts), K, alpha, 4, 3, cross_check=False)

"""Calls that run short of device memory half way: the allocations after the k-th fail, once or from
there on (a hook on the host; no memory is filled). What the library documents as another way to
the same result takes that way, everything else ends with TS_ERR_OOM, and the next call is whole."""
import numpy as np
import pytest

import oracle
from paper_1410_2698_gb300 import _lib, api
from paper_1410_2698_gb300.workloads import Segments
from tests import parity
from tests.cases import random_segments

pytestmark = pytest.mark.gpu

ALL = 1 << 40
TS_ERR_OOM = 2


@pytest.mark.parametrize("n", [300, 9000, 2200000])
@pytest.mark.parametrize("count", [1, ALL])
def test_sorted_rows_reach_the_host(n, count):
    """Rows sorted on the device, or by the host when any of its allocations fails."""
    m = np.zeros((n, 8))
    m[:, 7] = 1.0 + np.arange(n) / n
    idx = api.ts_build_index(Segments.from_matrix(m), kind="brute")
    res = api.ts_search(idx, Segments.from_matrix(m[-1:]), 1.0, 0.0, 5.0)
    assert res.count == n
    for k in range(12):
        api.ts_debug_fail_allocs(k, count)
        try:
            got = res.to_host(sort=True)
        finally:
            api.ts_debug_fail_allocs(0, 0)
        assert np.array_equal(got["e_idx"], np.arange(n)), k
        assert np.all(got["q_idx"] == 0) and np.all(got["t_in"] == 0)
        assert np.array_equal(got["t_out"], np.minimum(m[:, 7], m[-1, 7]))
    res.free()
    idx.free()


@pytest.mark.parametrize("kind", ["temporal", "spatial"])
@pytest.mark.parametrize("nq,d", [(40, 1.0), (40, 9.0), (3000, 1.0)])
def test_searches_take_the_stepwise_path(kind, nq, d):
    """A plain search in one go (query columns in place and copied, rows as guessed and more) with one
    allocation failing: the stepwise path answers. With all failing from the k-th on: TS_ERR_OOM."""
    rng = np.random.default_rng(41)
    db = random_segments(rng, 5000, box=20.0)
    q = random_segments(rng, nq, box=20.0)
    idx = api.ts_build_index(db, kind=kind)
    ref = oracle.search(db, q, 0.0, 12.0, d)
    for count in (1, ALL):
        failed = 0
        for k in range(24):
            api.ts_debug_fail_allocs(k, count)
            try:
                res = api.ts_search(idx, q, d, 0.0, 12.0)
            except _lib.TsError as e:
                assert e.status == TS_ERR_OOM, str(e)
                failed += 1
                continue
            finally:
                api.ts_debug_fail_allocs(0, 0)
            assert res.stats["n_queries"] == nq and res.stats["n_hits"] == res.count
            parity.compare(res.to_host(sort=True), ref, db, q, 0.0, 12.0, d)
            res.free()
        assert failed == 0 if count == 1 else 0 < failed < 24
    idx.free()

"""Calls that run short of device memory half way: the allocations after the k-th fail, once or from
there on (a hook on the host; no memory is filled). What the library documents as another way to
the same result takes that way, everything else ends with TS_ERR_OOM, and the next call is whole."""
import numpy as np
import pytest

from paper_1410_2698_gb300 import api
from paper_1410_2698_gb300.workloads import Segments

pytestmark = pytest.mark.gpu

ALL = 1 << 40


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

"""The radix sort at the edges of its forms (one block up to 2048 keys, tiles of 4096 that add up
the histograms themselves up to 2M keys, scanned histograms above) seen through the index's order
by start time: stable, for start times that differ in all bits, in few, and in none."""
import numpy as np
import pytest

from paper_1410_2698_gb300 import api
from paper_1410_2698_gb300.workloads import Segments

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 2047, 2048, 2049, 4097, 70001, 2097152, 2097153])
@pytest.mark.parametrize("times", ["any", "signed", "integers", "one"])
def test_entries_in_start_order(n, times):
    rng = np.random.default_rng(n)
    t0 = {"any": lambda: rng.uniform(0, 100, n), "signed": lambda: rng.normal(size=n) * 1e3,
          "integers": lambda: rng.integers(-3, 9, n) * 1.0,
          "one": lambda: np.full(n, 0.0)}[times]()
    if times == "integers":
        t0[t0 == 0.0] *= rng.choice([1.0, -1.0], (t0 == 0.0).sum())  # -0.0 is 0.0
    p = np.zeros((n, 3))
    m = np.concatenate([p, t0[:, None], p + 1.0, t0[:, None] + 1.0], axis=1)
    idx = api.ts_build_index(Segments.from_matrix(m), kind="temporal", t_bins=7)
    assert np.array_equal(api.ts_index_export(idx, "perm"), np.argsort(t0, kind="stable"))

"""The lookup tables of query preparation around the size up to which they are copied into shared
memory: 20 B a bin and 4, and with subbins 24 B each and 24 more; searches, schedules and plans on
indexes on both sides of it, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1410_2698_gb300 import api
from tests import parity
from tests.cases import random_segments

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,bins", [("temporal", m) for m in (2443, 2444, 2445, 2457, 2458)] +
                         [("spatiotemporal", m) for m in (2423, 2424, 2425, 2437, 2438)])
def test_searches_around_the_limit(kind, bins):
    rng = np.random.default_rng(bins)
    db = random_segments(rng, 4000, box=60.0, t_range=(0.0, 900.0))
    q = random_segments(rng, 60, box=60.0, t_range=(0.0, 900.0), max_dur=300.0)
    kw = {"sub_bins": 16} if kind == "spatiotemporal" else {}
    idx = api.ts_build_index(db, kind=kind, t_bins=bins, **kw)
    if kw:
        assert list(idx.info()["sub_bins"]) == [16, 16, 16]
    ref = oracle.search(db, q, 100.0, 800.0, 4.0)
    assert ref["q_idx"].size > 0
    res = api.ts_search(idx, q, 4.0, 100.0, 800.0)
    parity.compare(res.to_host(sort=True), ref, db, q, 100.0, 800.0, 4.0)
    _, lo, hi = api.ts_schedule(idx, q, 4.0, 100.0, 800.0)
    assert res.stats["n_tests"] == int((hi - lo).sum())
    plan = api.BatchPlan(idx, max_requests=1, max_queries=q.n, max_rows=res.count + 1)
    plan.run([(q, 4.0, 100.0, 800.0)])
    assert plan.wait()["rows"] == res.count
    plan.free()

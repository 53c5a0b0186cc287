"""How many hits the count pass keeps: a caller's scratch_rows exactly, the default all that a plan has
rows for, with hits spread over all warps a few each (a warp's slots taken in advance stay empty)."""
import ctypes

import numpy as np
import pytest

from paper_1410_2698_gb300 import _lib, api
from tests.cases import random_segments

pytestmark = pytest.mark.gpu


def _once(plan):
    once = ctypes.c_int32(-1)
    _lib.check(_lib.load().ts_debug_batch_swept_once(plan.handle, ctypes.byref(once)))
    return once.value


@pytest.mark.parametrize("kind", ["temporal", "spatial", "brute"])
@pytest.mark.parametrize("nq,d", [(40, 1.0), (6000, 0.7), (6000, 4.0)])
def test_hits_kept(kind, nq, d):
    rng = np.random.default_rng(nq)
    db = random_segments(rng, 30000, box=60.0)
    q = random_segments(rng, nq, box=60.0)
    idx = api.ts_build_index(db, kind=kind)
    ref = api.ts_search(idx, q, d, 0.0, 12.0)
    want, n = ref.to_host(), ref.count
    assert n > 20
    for scratch, once in ((0, 1), (n, 1), (n + 1, 1), (2 * n, 1), (n - 1, 0), (n // 2, 0), (1, 0)):
        plan = api.BatchPlan(idx, max_requests=1, max_queries=nq, max_rows=n, scratch_rows=scratch,
                             max_units=512 * nq if kind == "spatial" else 0)
        for _ in range(2):
            plan.run([(q, d, 0.0, 12.0)])
            st = plan.wait()
            assert not st["overflow"] and st["rows"] == n and _once(plan) == once, scratch
        got = plan.request_to_host(0)
        for k, v in want.items():
            assert np.array_equal(got[k], v), (scratch, k)
        plan.free()
    idx.free()

"""Tiles and chunks listed for the pair kernel by their bounding records: sizes around the chunk
(64), the tile and the group (32), on databases where the Morton order has nothing to tell apart
(a point, a line, a plane) and where it has, against the oracle, for every kind of index."""
import numpy as np
import pytest

import oracle
from paper_1410_2698_gb300 import api
from paper_1410_2698_gb300.workloads import Segments
from tests import parity
from tests.cases import random_segments

pytestmark = pytest.mark.gpu


def _flat(rng, n, axes):
    """Random segments of a box whose extent is zero but in the first `axes` axes."""
    m = random_segments(rng, n, box=40.0, t_range=(0, 20), max_len=2.0).as_matrix()
    for k in range(axes, 3):
        m[:, k] = m[:, 4 + k] = 7.0
    return Segments.from_matrix(m)


@pytest.mark.parametrize("kind", ["temporal", "spatiotemporal", "spatial", "brute"])
@pytest.mark.parametrize("n,nq", [(1, 1), (63, 33), (65, 1), (2049, 31), (20000, 700)])
@pytest.mark.parametrize("axes", [0, 1, 3])
def test_rows_equal_the_oracle(kind, n, nq, axes):
    rng = np.random.default_rng(1000 * axes + n)
    db, q = _flat(rng, n, axes), _flat(rng, nq, axes)
    d = 0.5 if axes < 3 else 3.0
    ref = oracle.search(db, q, 2.0, 19.0, d)
    idx = api.ts_build_index(db, kind=kind)
    res = api.ts_search(idx, q, d, 2.0, 19.0)
    parity.compare(res.to_host(sort=True), ref, db, q, 2.0, 19.0, d)
    # candidates are counted where the schedule made them, listed or not
    if kind != "spatial":
        _, lo, hi = api.ts_schedule(idx, q, d, 2.0, 19.0)
        assert res.stats["n_tests"] == int((hi - lo).sum())


@pytest.mark.parametrize("kind", ["temporal", "spatiotemporal"])
def test_far_queries_and_many_requests(kind):
    """Queries outside the database's extents (their Morton cell is the nearest one) beside queries
    inside, in so many requests that little of the sort key is left for the place."""
    rng = np.random.default_rng(5)
    db = random_segments(rng, 5000, box=40.0, t_range=(0, 20))
    m = random_segments(rng, 300, box=40.0, t_range=(0, 20)).as_matrix()
    m[::3, [0, 1, 2, 4, 5, 6]] += np.array([1e6, -1e5, 50.0] * 2)
    q = Segments.from_matrix(m)
    idx = api.ts_build_index(db, kind=kind)
    reqs = [(q.take(np.arange(r % 7, 300, 7)), 2.0, 0.0, 20.0 - r % 3) for r in range(70)]
    for (qr, d, ts, te), res in zip(reqs, api.ts_search_batch(idx, reqs)):
        parity.compare(res.to_host(sort=True), oracle.search(db, qr, ts, te, d), db, qr, ts, te, d)


@pytest.mark.parametrize("tile", [64, 192, 512])
@pytest.mark.parametrize("scratch", [0, 300])
def test_runs_of_tiles(tile, scratch):
    """So many tiles that a listed entry holds a run of them (16,000 queries against all of 400,000
    entries in tiles of 64 are 3.1M), with all hits kept for placement and with the flagged tiles
    of the runs swept again: the rows and their order are the plain search's."""
    rng = np.random.default_rng(9)
    db = random_segments(rng, 400000, box=300.0)
    q = random_segments(rng, 16000, box=300.0)
    idx = api.ts_build_index(db, kind="brute")
    ref = api.ts_search(idx, q, 1.0, 0.0, 12.0)
    want = ref.to_host()
    plan = api.BatchPlan(idx, max_requests=1, max_queries=q.n, max_rows=ref.count + 10,
                         tile_records=tile, max_tiles=4 << 20, scratch_rows=scratch)
    plan.run([(q, 1.0, 0.0, 12.0)])
    st = plan.wait()
    assert not st["overflow"] and st["rows"] == ref.count > 300
    got = plan.request_to_host(0)
    for k in ("q_idx", "e_idx", "t_in", "t_out"):
        assert np.array_equal(got[k], want[k]), k
    plan.free()

"""The order of a bin's entries: by x where the occupied bins hold 4,096 entries or fewer on average,
along the Morton curve where they hold more. Databases on both sides of the line, bins of very
different sizes and mostly empty ones, with and without extents to tell apart, queries inside and
outside, plain and in a batch, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1410_2698_gb300 import api
from paper_1410_2698_gb300.workloads import Segments
from tests import parity
from tests.cases import random_segments

pytestmark = pytest.mark.gpu


def _db(n, times, axes):
    """n segments that start at one of `times` (one of them most often), flat but in `axes` axes."""
    rng = np.random.default_rng(n)
    m = random_segments(rng, n, box=80.0, max_len=2.0).as_matrix()
    k = rng.integers(0, len(times), n)
    k[: len(times)] = np.arange(len(times))
    m[:, 3] = np.asarray(times)[k]
    m[:, 7] = m[:, 3] + 1.0
    for a in range(axes, 3):
        m[:, a] = m[:, 4 + a] = 7.0
    return Segments.from_matrix(m)


@pytest.mark.parametrize("kind", ["temporal", "spatiotemporal"])
@pytest.mark.parametrize("n,bins,times", [(4096, 1, [0.0]), (4097, 1, [0.0]),
                                          (3 * 4096, 40, [0.0, 3.0, 9.0]),
                                          (3 * 4096 + 1, 40, [0.0, 3.0, 9.0]),
                                          (60000, 7, [0.0, 0.5, 9.0])])
@pytest.mark.parametrize("axes", [0, 1, 3])
def test_rows_on_both_sides_of_the_line(kind, n, bins, times, axes):
    db = _db(n, times, axes)
    rng = np.random.default_rng(7)
    m = random_segments(rng, 400 if axes == 3 else 20, box=80.0, t_range=(-1.0, 10.0)).as_matrix()
    m[::5, [0, 1, 2, 4, 5, 6]] += np.array([1e5, -90.0, 50.0] * 2)
    for a in range(axes, 3):
        m[:, a] = m[:, 4 + a] = 7.0
    q = Segments.from_matrix(m)
    idx = api.ts_build_index(db, kind=kind, t_bins=bins)
    d = 2.0 if axes == 3 else 0.5
    ref = oracle.search(db, q, 0.2, 9.6, d)
    assert ref["q_idx"].size > 0
    parity.compare(api.ts_search(idx, q, d, 0.2, 9.6).to_host(sort=True), ref, db, q, 0.2, 9.6, d)
    reqs = [(q, d, 0.2, 9.6), (q.take(np.arange(0, q.n, 3)), d / 2, 0.0, 5.0)]
    for (qr, dr, ts, te), res in zip(reqs, api.ts_search_batch(idx, reqs)):
        parity.compare(res.to_host(sort=True), oracle.search(db, qr, ts, te, dr), db, qr, ts, te, dr)
    info = api.ts_index_get_info(idx)
    tidx = oracle.temporal_index(db.t0, db.t1, info["t_bins"])
    for f in ("perm", "bin_off"):
        np.testing.assert_array_equal(api.ts_index_export(idx, f), tidx[f])

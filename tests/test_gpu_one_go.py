"""Plain searches enqueued in one go on guessed capacities: guesses that hold and guesses that do
not (cell runs, tiles, rows, queries above what one go takes), host queries read in place and
copied, more searches at a time than there are slots; every result against the oracle."""
import threading

import numpy as np
import pytest

import oracle
from paper_1410_2698_gb300 import _lib, api
from paper_1410_2698_gb300.workloads import Segments
from tests import parity
from tests.cases import random_segments

pytestmark = pytest.mark.gpu


def _check(idx, db, q, d, ts, te, device=False):
    import torch
    qq = q
    if device:
        qq = [torch.from_numpy(np.ascontiguousarray(c)).cuda() for c in q.arrays()]
    res = api.ts_search(idx, qq, d, ts, te)
    ref = oracle.search(db, q, ts, te, d)
    parity.compare(res.to_host(sort=True), ref, db, q, ts, te, d)
    assert res.count == ref["q_idx"].size == res.stats["n_hits"]
    assert res.stats["n_queries"] == q.n and res.stats["ms_count_pass"] > 0
    return res.count


@pytest.mark.parametrize("nq", [1, 1024, 1025, 20000])
@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("kind", ["temporal", "spatiotemporal", "spatial", "brute"])
def test_query_counts(kind, device, nq):
    rng = np.random.default_rng(nq)
    db = random_segments(rng, 3000, box=30.0)
    q = random_segments(rng, nq, box=30.0)
    _check(api.ts_build_index(db, kind=kind), db, q, 1.0, 1.0, 9.0, device)


def test_more_rows_than_asked_for_and_none():
    rng = np.random.default_rng(2)
    db = random_segments(rng, 5000, box=5.0)
    q = random_segments(rng, 40, box=5.0)
    idx = api.ts_build_index(db, kind="temporal")
    assert _check(idx, db, q, 4.0, 0.0, 12.0) > 64 + 8 * q.n
    assert _check(idx, db, q, 4.0, 50.0, 60.0) == 0
    few = api.ts_search(idx, q, 4.0, 0.0, 12.0, max_results=7)
    assert few.status == 4 and few.count > 7 and few.device_arrays() == (None,) * 4


def test_more_cell_runs_than_guessed():
    """Queries across the whole grid, far longer than any entry: hundreds of runs of cells each,
    where a handful is guessed."""
    rng = np.random.default_rng(3)
    db = random_segments(rng, 4000, box=100.0)
    q = random_segments(rng, 200, box=100.0, max_len=90.0)
    idx = api.ts_build_index(db, kind="spatial", grid_cells=64)
    assert int(api.ts_schedule(idx, q, 1.0, 0.0, 12.0)[1].sum()) > 49 * q.n + 1024
    _check(idx, db, q, 1.0, 0.0, 12.0)


@pytest.mark.parametrize("d", [0.2, 5.0, 60.0])
def test_distances_of_a_part_of_a_cell_to_all_cells(d):
    rng = np.random.default_rng(8)
    db = random_segments(rng, 3000, box=50.0)
    q = random_segments(rng, 70, box=50.0)
    _check(api.ts_build_index(db, kind="spatial"), db, q, d, 0.0, 12.0)


def test_more_tiles_than_guessed():
    """3,000 query segments as long as 500 entries, one after another in a group's 32 bins' worth of
    entries: their ranges take all 977 tiles where a few bins' are guessed."""
    rng = np.random.default_rng(4)
    db = random_segments(rng, 250000, box=400.0, t_range=(0.0, 500.0), max_dur=1.0)
    m = random_segments(rng, 3000, box=400.0).as_matrix()
    m[:, 3], m[:, 7] = 0.0, 501.0
    q = Segments.from_matrix(m)
    idx = api.ts_build_index(db, kind="temporal")
    _check(idx, db, q, 2.0, 0.0, 501.0)
    assert api.ts_search(idx, q, 2.0, 0.0, 501.0).stats["n_tiles"] > 50 * 95 + 65536


def test_more_queries_than_one_go_takes():
    rng = np.random.default_rng(5)
    db = random_segments(rng, 2000, box=60.0)
    q = random_segments(rng, 65537, box=60.0)
    _check(api.ts_build_index(db, kind="spatiotemporal"), db, q, 0.5, 0.0, 12.0, True)


def test_invalid_queries_and_columns():
    import ctypes
    rng = np.random.default_rng(6)
    db = random_segments(rng, 500)
    idx = api.ts_build_index(db, kind="spatial")
    m = random_segments(rng, 30).as_matrix()
    m[7, 2] = np.nan
    with pytest.raises(_lib.TsError, match="invalid query segment"):
        api.ts_search(idx, Segments.from_matrix(m), 1.0, 0.0, 9.0)
    s, keep = api.make_segments(random_segments(rng, 30))
    s.y1 = None
    qp = _lib.ts_query_params(1.0, 0.0, 9.0, 0)
    out = ctypes.c_void_p()
    assert _lib.load().ts_search(idx.handle, ctypes.byref(s), ctypes.byref(qp), None,
                                 ctypes.byref(out)) == 1
    assert "NULL query column" in api.ts_last_error()
    _check(idx, db, random_segments(rng, 30), 1.0, 0.0, 9.0)


def test_threads_and_streams():
    """24 threads with a stream each, 16 slots: the others wait for sizes step by step."""
    import torch
    rng = np.random.default_rng(7)
    db = random_segments(rng, 4000, box=20.0)
    idx = api.ts_build_index(db, kind="spatial")
    sets = [random_segments(rng, 50 + 13 * k, box=20.0) for k in range(24)]
    refs = [oracle.search(db, q, 0.0, 12.0, 2.0) for q in sets]
    errors = []

    def work(k):
        try:
            s = torch.cuda.Stream()
            for _ in range(6):
                got = api.ts_search(idx, sets[k], 2.0, 0.0, 12.0, stream=s.cuda_stream)
                parity.compare(got.to_host(stream=s.cuda_stream, sort=True), refs[k], db, sets[k], 0.0, 12.0,
                               2.0)
        except Exception as e:  # noqa: BLE001
            errors.append((k, e))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(24)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


@pytest.mark.parametrize("n", [1, 2729, 2730, 2731, 9000])
def test_rows_to_host(n):
    """Rows through a slot (up to 2,730) and by four copies are the device's rows."""
    m = np.zeros((n, 8))
    m[:, 7] = 1.0 + np.arange(n) / n
    idx = api.ts_build_index(Segments.from_matrix(m), kind="temporal")
    res = api.ts_search(idx, Segments.from_matrix(m[:1]), 1.0, 0.0, 5.0)
    assert res.count == n
    host = res.to_host()
    assert np.array_equal(np.sort(host["e_idx"]), np.arange(n))
    assert np.all(host["q_idx"] == 0) and np.all(host["t_in"] == 0) and np.all(host["t_out"] == 1)
    lib = _lib.load()
    only = np.empty(n, np.uint32)  # a destination of its own, the others left out
    _lib.check(lib.ts_result_copy_to_host(res.handle, None, only.ctypes.data, None, None, None))
    assert np.array_equal(only, host["e_idx"])


@pytest.mark.parametrize("nq,box", [(1, 4.0), (3, 8.0), (40, 12.0), (300, 20.0), (2000, 12.0)])
@pytest.mark.parametrize("kind", ["spatiotemporal", "spatial"])
def test_rows_sorted_on_the_device(nq, box, kind):
    """Rows by (query, entry) as numpy sorts them: few (sorted by the host, or through a slot) and
    many, of a search and of a batch, also one field alone."""
    rng = np.random.default_rng(nq)
    db = random_segments(rng, 3000, box=box)
    q = random_segments(rng, nq, box=box)
    idx = api.ts_build_index(db, kind=kind)
    lib = _lib.load()
    for res in (api.ts_search(idx, q, 2.0, 0.0, 12.0),
                api.ts_search_batch(idx, [(q, 1.0, 0.0, 12.0), (q, 2.0, 0.0, 12.0)])[1]):
        rows = res.to_host()
        order = np.lexsort((rows["e_idx"], rows["q_idx"]))
        got = res.to_host(sort=True)
        assert rows["q_idx"].size == res.count > 0
        for k, v in rows.items():
            assert np.array_equal(got[k], v[order]), k
        only = np.empty(res.count)
        _lib.check(lib.ts_result_copy_sorted_to_host(res.handle, None, None, None,
                                                     only.ctypes.data, None))
        assert np.array_equal(only, rows["t_out"][order])


@pytest.mark.parametrize("kind", ["temporal", "spatiotemporal"])
def test_points_over_the_whole_interval(kind):
    """3,000 fixed points meet all of the 2,000 bins: they take the kernels of 1,000 points and those of
    a sort of more than one block, not a second search step by step."""
    rng = np.random.default_rng(12)
    db = random_segments(rng, 200000, box=300.0, t_range=(0.0, 1000.0), max_dur=0.4)
    idx = api.ts_build_index(db, kind=kind, t_bins=2000)
    took = []
    for n in (1000, 3000):
        p = rng.uniform(0.0, 300.0, (n, 3))
        before = api.ts_kernel_launches()
        res = api.ts_search_points(idx, p[:, 0], p[:, 1], p[:, 2], 1.0, -5.0, 2000.0)
        took.append(api.ts_kernel_launches() - before)
        m = np.column_stack([p, np.full(n, -5.0), p, np.full(n, 2000.0)])
        ref = oracle.search(db, Segments.from_matrix(m), -5.0, 2000.0, 1.0)
        got = res.to_host(sort=True)
        assert ref["q_idx"].size > 0
        for k in ("q_idx", "e_idx"):
            assert np.array_equal(got[k], ref[k])
    assert took[1] <= took[0] + 10, took

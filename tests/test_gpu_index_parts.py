"""Subbins and cells found from the boundary tables, where the first guess in FP32 is poor:
coordinates far from the origin, extents of a few ulps, huge and tiny scales, one point; against
the oracle's arrays. A bin whose latest end is found by one atomic for a warp, and by many."""
import numpy as np
import pytest

import oracle
from paper_1410_2698_gb300 import api
from paper_1410_2698_gb300.workloads import Segments
from tests.cases import random_segments

pytestmark = pytest.mark.gpu

SHAPES = {"plain": (1.0, 0.0), "far": (1.0, 1e9), "ulps": (1e-9, 1e6), "huge": (1e200, 0.0),
          "tiny": (1e-200, 0.0), "point": (0.0, 3.0)}


def _db(shape, n):
    scale, shift = SHAPES[shape]
    rng = np.random.default_rng(31)
    m = random_segments(rng, n, box=10.0, t_range=(0.0, 40.0), max_len=1.0).as_matrix()
    m[:, [0, 1, 2, 4, 5, 6]] = m[:, [0, 1, 2, 4, 5, 6]] * scale + shift
    return Segments.from_matrix(m)


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("n", [33, 5000])
def test_subbins(shape, n):
    db = _db(shape, n)
    m = 50
    idx = api.ts_build_index(db, kind="spatiotemporal", t_bins=m, sub_bins=16)
    info = api.ts_index_get_info(idx)
    ref = oracle.temporal_index(db.t0, db.t1, m)
    for f in ("perm", "bin_start", "bin_end", "bin_off"):
        np.testing.assert_array_equal(api.ts_index_export(idx, f), ref[f])
    for dim, (a, b) in enumerate(((db.x0, db.x1), (db.y0, db.y1), (db.z0, db.z1))):
        lo, hi = np.minimum(a, b)[ref["perm"]], np.maximum(a, b)[ref["perm"]]
        ids, off = oracle.st_dim(lo, hi, ref["bin_of"], m, info["sub_lo"][dim],
                                 info["sub_w"][dim], info["sub_bins"][dim])
        np.testing.assert_array_equal(api.ts_index_export(idx, "st_ids", dim), ids)
        np.testing.assert_array_equal(api.ts_index_export(idx, "st_off", dim), off)


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("g", [1, 7, 200])
def test_cells(shape, g):
    db = _db(shape, 3000)
    idx = api.ts_build_index(db, kind="spatial", grid_cells=g)
    info = api.ts_index_get_info(idx)
    perm = oracle.temporal_index(db.t0, db.t1, 1)["perm"]
    low = [np.minimum(a, b)[perm] for a, b in ((db.x0, db.x1), (db.y0, db.y1), (db.z0, db.z1))]
    A, off = oracle.grid1(low, g, info["grid_lo"], info["grid_w"])
    np.testing.assert_array_equal(api.ts_index_export(idx, "grid_a"), A)
    np.testing.assert_array_equal(api.ts_index_export(idx, "grid_off"), off)


def test_an_index_in_the_pool_is_given_back():
    """Building and freeing an index again and again holds no more device memory."""
    import torch
    db = _db("plain", 200000)
    used = []
    for _ in range(4):
        idx = api.ts_build_index(db, kind="spatiotemporal")
        idx.free()
        torch.cuda.synchronize()
        used.append(torch.cuda.mem_get_info()[0])
    assert max(used[1:]) - min(used[1:]) < (1 << 20)


def test_freed_indexes_leave_a_bound():
    """What freed indexes leave in the pool is bounded for all together (512 MB, and a few blocks of
    memory that the pool gives back whole), for many of less than that and for one of more."""
    import torch
    rng = np.random.default_rng(6)
    db = random_segments(rng, 1000000, box=200.0, max_len=1.0)
    idx = api.ts_build_index(db, kind="spatiotemporal")
    size = idx.info()["device_bytes"]
    idx.free()
    torch.cuda.synchronize()
    room = torch.cuda.mem_get_info()[0]
    many = int(2e9 // size) + 1
    assert size < (512 << 20)
    held = [api.ts_build_index(db, kind="spatiotemporal") for _ in range(many)]
    for idx in held:
        idx.free()
    torch.cuda.synchronize()
    assert room - torch.cuda.mem_get_info()[0] < (640 << 20)
    big = Segments.from_matrix(np.tile(db.as_matrix(), (6, 1)))
    idx = api.ts_build_index(big, kind="spatiotemporal")
    size = idx.info()["device_bytes"]
    assert size > (700 << 20)
    alive = torch.cuda.mem_get_info()[0]
    idx.free()
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] - alive > size - (640 << 20)
    idx = api.ts_build_index(db, kind="spatiotemporal")
    q = db.take(np.arange(50))
    assert api.ts_search(idx, q, 0.5, 0.0, 13.0).count >= 50
    idx.free()

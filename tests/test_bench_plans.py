"""How bench.py sizes its batch plans: room for the tiles of any record count from the plain searches'
count in tiles of 256, and a plan whose first run does not fit is built again with the count the
device reported, or given up."""
import numpy as np
import pytest

import bench
from paper_1410_2698_gb300 import autotune


@pytest.mark.parametrize("tile", [0, 64, 192] + autotune.TILES)
def test_room_for_tiles_of_any_size(tile):
    """Ranges of any length: no more tiles of `tile` records than the room made from the tiles of 256."""
    rng = np.random.default_rng(tile)
    for n in (rng.integers(1, 300, 400000), rng.integers(1, 40000, 100000), np.full(300000, 129)):
        plain = int(np.sum(-(-n // 256)))
        assert int(np.sum(-(-n // (tile or 256)))) <= bench.plan_tiles(plain, tile)


class _Plan:
    live = 0

    def __init__(self, tiles):
        self.tiles = tiles
        _Plan.live += 1

    def free(self):
        _Plan.live -= 1


def _run(need, rows_fit=True):
    def run(plan):
        over = need > plan.tiles or not rows_fit
        return {"overflow": over, "rows": 7, "stats": {"n_tiles": need}}
    return run


def test_a_plan_that_does_not_fit_is_built_again():
    _Plan.live = 0
    assert bench.fitting_plan(_Plan, _run(1000), 1000).tiles == 1000
    assert bench.fitting_plan(_Plan, _run(1000), 10).tiles >= 1000
    assert _Plan.live == 2  # the one that did not fit was freed
    with pytest.raises(RuntimeError, match="overflow"):
        bench.fitting_plan(_Plan, _run(1000, rows_fit=False), 2000)
    assert _Plan.live == 2


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["temporal", "spatiotemporal", "spatial"])
@pytest.mark.parametrize("tile", [64] + autotune.TILES)
def test_plans_of_any_tile_size_fit(kind, tile):
    """A plan of several requests in the room made from the plain searches of each."""
    from paper_1410_2698_gb300 import api, workloads
    w = workloads.tiny()
    idx = api.ts_build_index(w.db, kind=kind)
    plain = [api.ts_search(idx, w.queries, d, w.t_start, w.t_end) for d in (2.0, 8.0)]
    tiles = sum(r.stats["n_tiles"] for r in plain)
    reqs = [(w.queries, d, w.t_start, w.t_end) for d in (2.0, 8.0)]

    def make(room):
        return api.BatchPlan(idx, max_requests=2, max_queries=2 * w.queries.n, tile_records=tile,
                             max_rows=sum(r.count for r in plain) + 1, max_tiles=room,
                             max_units=512 * w.queries.n if kind == "spatial" else 0)

    def run(plan):
        plan.run(reqs)
        return plan.wait()

    assert bench.plan_tiles(tiles, tile) >= tiles
    for room in (bench.plan_tiles(tiles, tile), 1):  # as the benchmark asks for it, and too little
        plan = bench.fitting_plan(make, run, room)
        st = run(plan)
        assert not st["overflow"] and st["rows"] == sum(r.count for r in plain)
        plan.free()
    idx.free()

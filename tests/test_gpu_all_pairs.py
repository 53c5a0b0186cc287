"""The no-allocation all-pairs search at the edges of its tiles (32 query segments x 1024 database
segments, in blocks of 32), with neighbours in the database near each other (blocks that no query
meets are skipped) and shuffled (every block is met), and for a database so large that a bounding
record covers more than one block; rows against the oracle, in tile order."""
import numpy as np
import pytest

import oracle
from paper_1410_2698_gb300 import api, workloads
from paper_1410_2698_gb300.workloads import Segments
from tests import parity
from tests.cases import random_segments

pytestmark = pytest.mark.gpu


def _search(db, q, d, ts, te, cap):
    import torch
    dev = [[torch.from_numpy(np.ascontiguousarray(c)).cuda() for c in s.arrays()] for s in (db, q)]
    out = [torch.zeros(cap, dtype=t, device="cuda")
           for t in (torch.int32, torch.int32, torch.float64, torch.float64)]
    st, n = api.ts_search_brute_noalloc(dev[0], dev[1], d, ts, te, *out)
    assert st == 0
    return {k: x[:n].cpu().numpy().astype(t) for k, x, t in
            zip(("q_idx", "e_idx", "t_in", "t_out"), out, (np.uint32, np.uint32, float, float))}


def _check(db, q, d, ts, te):
    ref = oracle.search(db, q, ts, te, d)
    got = _search(db, q, d, ts, te, ref["q_idx"].size + 8)
    tile = got["q_idx"].astype(np.int64) // 32 * (1 << 32) + got["e_idx"] // 1024
    assert np.all(np.diff(tile) >= 0)  # rows grouped by tile, in tile order
    order = np.lexsort((got["e_idx"], got["q_idx"]))
    parity.compare({k: v[order] for k, v in got.items()}, ref, db, q, ts, te, d)
    return ref["q_idx"].size


@pytest.mark.parametrize("nq,n", [(1, 1), (31, 33), (32, 1024), (33, 1025), (64, 1023), (65, 2049)])
@pytest.mark.parametrize("shuffled", [False, True])
def test_tile_edges(nq, n, shuffled):
    w = workloads.tiny()
    order = np.arange(w.db.n)
    if shuffled:
        order = np.random.default_rng(7).permutation(w.db.n)
    db = w.db.take(order[:n])
    q = w.queries.take(np.arange(nq))
    _check(db, q, 5.0, 2.0, 69.0)


def test_every_pair_passes_the_filters():
    """A tile whose 32 x 1024 pairs all reach the exact test (the longest list of pairs)."""
    rng = np.random.default_rng(3)
    db = random_segments(rng, 1100, box=1.0, t_range=(0, 1), max_len=0.5, max_dur=3.0)
    q = random_segments(rng, 40, box=1.0, t_range=(0, 1), max_len=0.5, max_dur=3.0)
    assert _check(db, q, 50.0, 0.0, 5.0) > 20000


@pytest.mark.parametrize("seg_per", [1, 400])
def test_bounding_records_of_more_than_one_block(seg_per):
    """4,000,000 database segments: the bounding records cover 64 segments each."""
    rng = np.random.default_rng(5)
    n = 4_000_000
    if seg_per == 1:  # no two neighbours near each other
        db = random_segments(rng, n, box=1000.0, t_range=(0, 100))
    else:
        pos, t = workloads._random_walk(rng, n // seg_per, seg_per + 1, (0.0, 1000.0),
                                        (0.0, 100.0), 2.0)
        db = workloads.samples_to_segments(pos, t)
    q = Segments.from_matrix(db.as_matrix()[rng.choice(n, 45, replace=False)])
    assert _check(db, q, 10.0, 0.0, 500.0) >= 45

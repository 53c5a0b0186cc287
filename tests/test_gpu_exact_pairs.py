"""The exact test in pairs of FP32 values where it can go wrong: space and time scaled by powers of
two inside and outside its range, separations at the threshold, tangent passes, no relative
motion, windows of every length, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1410_2698_gb300 import api
from paper_1410_2698_gb300.workloads import Segments
from tests import parity
from tests.cases import random_segments, segset

pytestmark = pytest.mark.gpu


def _both(db, q, d, ts, te):
    """Rows of the indexed and of the all-pairs search, each compared with the oracle."""
    import torch
    ref = oracle.search(db, q, ts, te, d)
    got = api.ts_search(api.ts_build_index(db, kind="brute"), q, d, ts, te).to_host(sort=True)
    out = parity.compare(got, ref, db, q, ts, te, d)
    dev = [[torch.from_numpy(np.ascontiguousarray(c)).cuda() for c in s.arrays()] for s in (db, q)]
    rows = [torch.zeros(ref["q_idx"].size + 64, dtype=t, device="cuda")
            for t in (torch.int32, torch.int32, torch.float64, torch.float64)]
    st, n = api.ts_search_brute_noalloc(dev[0], dev[1], d, ts, te, *rows)
    assert st == 0
    flat = {k: x[:n].cpu().numpy().astype(t) for k, x, t in
            zip(("q_idx", "e_idx", "t_in", "t_out"), rows, (np.uint32, np.uint32, float, float))}
    order = np.lexsort((flat["e_idx"], flat["q_idx"]))
    for k, v in flat.items():
        assert np.array_equal(v[order], got[k]), k
    return ref, out


@pytest.mark.parametrize("space", [-40, -21, -19, 0, 17, 40])
@pytest.mark.parametrize("time", [-40, -21, 0, 19, 40])
def test_scales(space, time):
    """The same pairs at scales of space and time inside, at the ends of and outside the range of
    the FP32 pairs: powers of two change no rounding, so neither the rows nor (scaled) times."""
    rng = np.random.default_rng(17)
    db = random_segments(rng, 600, box=10.0, stationary_frac=0.2)
    m = random_segments(rng, 100, box=10.0, stationary_frac=0.2).as_matrix()
    m[::10] = db.as_matrix()[:100:10]  # the entry itself: no separation, no relative motion
    f = np.array([2.0 ** space] * 3 + [2.0 ** time]) [[0, 1, 2, 3, 0, 1, 2, 3]]
    dbs, qs = (Segments.from_matrix(x * f) for x in (db.as_matrix(), m))
    ref, out = _both(dbs, qs, 2.0 * 2.0 ** space, 0.0, 12.0 * 2.0 ** time)
    plain = oracle.search(db, Segments.from_matrix(m), 0.0, 12.0, 2.0)
    assert np.array_equal(ref["q_idx"], plain["q_idx"]) and ref["q_idx"].size > 0
    assert out["exempt"] == 0


def test_separations_at_the_threshold():
    """Resting points exactly d apart (hits, for the whole window), an ulp more and less, and passes
    whose closest separation is d times 1 +- 2^-k."""
    q = segset([[0, 0, 0, 0, 0, 0, 0, 1]])
    rows, want = [], []
    for x, y, z in ((3, 4, 0), (0, -5, 0), (4, 0, -3), (0, 3, 4)):
        for s, hit in ((1.0, True), (1.0 + 2.0 ** -45, False), (1.0 - 2.0 ** -45, True)):
            rows.append([x * s, y * s, z * s, 0, x * s, y * s, z * s, 1])
            want.append(hit)
    for k in range(4, 29):
        for sign, hit in ((1, False), (-1, True)):
            s = 5.0 * (1.0 + sign * 2.0 ** -k)
            rows.append([-2, s, 0, 0, 2, s, 0, 1])
            want.append(hit)
    ref, out = _both(segset(rows), q, 5.0, 0.0, 1.0)
    assert out["exempt"] == 0
    assert np.array_equal(np.isin(np.arange(len(want)), ref["e_idx"]), np.array(want))


@pytest.mark.parametrize("window", [1e-9, 1e-4, 1.0])
def test_windows(window):
    """Query intervals far shorter than the segments: roots beyond the window at both ends."""
    rng = np.random.default_rng(23)
    db = random_segments(rng, 2000, box=8.0, t_range=(4.0, 5.0), max_len=6.0)
    q = random_segments(rng, 150, box=8.0, t_range=(4.0, 5.0), max_len=6.0)
    ref, _ = _both(db, q, 1.5, 5.5, 5.5 + window)
    assert ref["q_idx"].size > 0


@pytest.mark.parametrize("end", ["in", "out"])
@pytest.mark.parametrize("near", ["start", "end"])
def test_roots_at_the_ends_of_the_window(end, near):
    """Entries that come within d (in) or leave (out) within two FP32 ulps of the ends of windows whose
    lengths have 53 random bits, on both sides of them: the pairs' high parts alone do not order a
    root and the window's end. One pair per place of a lattice, so a query meets one entry."""
    rng = np.random.default_rng(29)
    n, d = 15 ** 3, 1.0
    place = 16.0 * np.stack(np.meshgrid(*[np.arange(15.0)] * 3), axis=-1).reshape(n, 3)
    T = rng.uniform(0.1, 2.0, n)
    root = rng.uniform(-2, 2, n) * np.spacing(T.astype(np.float32)).astype(float)
    if near == "end":
        root += T
    u, v = rng.normal(size=(2, n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    # the separation grows at the root (out) or shrinks (in)
    v *= np.where((np.sum(u * v, axis=1) > 0) == (end == "out"), 1.0, -1.0)[:, None]
    p0 = place + d * u - v * (root + 1.0)[:, None]  # at time -1
    q = Segments.from_matrix(np.column_stack([place, np.zeros(n), place, T]))
    db = Segments.from_matrix(np.column_stack([p0, np.full(n, -1.0), p0 + 4.0 * v, np.full(n, 3.0)]))
    ref, out = _both(db, q, d, -1.0, 3.0)
    assert n // 4 < ref["q_idx"].size <= n and out["worst_out"] < 1e-9

"""What a user of the library has it do, as timed cases.

Every case goes through the public entry points of ``paper_1410_2698_gb300.api`` (or, for the device
rows of a plan, the C call behind them) on the repository's own kinds of trajectories: random walks,
a dense cube, and a two-cluster merger (``workloads.py`` has the recipes; the same ones are drawn
here on the GPU, from the case's seed).

A search's rows come in the library's own order, which is fixed but not a promise, and a program that
needs an order sorts them by (query, entry). Cases with rows = "sorted" do that, on the device or
with the binding's own ``sort=True`` on the host; the others hand the rows on as they come. A program
has row arrays of its own, with room for more rows than it expects: outputs are these arrays (or a
plan's own), zero past the rows.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1410_2698_gb300 import _lib, api

DEV = "cuda"


def listed():
    return [
        # smallest call: one trajectory of 20 segments against a small database, host arrays in,
        # sorted host rows out (an interactive query)
        dict(name="one-trajectory", form="search", data="walk", traj=1000, samples=21, box=100.0,
             sigma=1.0, spread=50.0, qtraj=1, kind="temporal", d="5", queries="host",
             rows="sorted"),
        # an ordinary search: 1% of a random-walk database against all of it, on the grid index
        dict(name="walk-search", form="search", data="walk", traj=2500, samples=401, box=1000.0,
             sigma=2.0, spread=100.0, qtraj=25, kind="spatial", d="10", queries="device",
             rows="device"),
        # many entries alive at once: 500 trajectories in a dense cube, temporal bins
        dict(name="dense-search", form="search", data="dense", traj=20000, samples=101, qtraj=500,
             kind="temporal", d="2", queries="device", rows="sorted"),
        # a search whose rows are many (hundreds per query segment), on the grid index
        dict(name="merger-search", form="search", data="merger", traj=10000, samples=201, qtraj=200,
             kind="spatial", d="5", queries="device", rows="device"),
        # fixed points over the whole interval (an odd number of them)
        dict(name="points-search", form="points", data="walk", traj=2500, samples=401, box=1000.0,
             sigma=2.0, spread=100.0, qtraj=777, kind="spatial", d="10", queries="device",
             rows="device"),
        # a resident plan for the same four distances again and again: queries from pinned host
        # memory, every row read back into pinned host memory
        dict(name="walk-plan", form="plan", data="walk", traj=2500, samples=401, box=1000.0,
             sigma=2.0, spread=100.0, qtraj=25, kind="spatial", d="1,5,10,25", queries="pinned",
             rows="host"),
        # a plan on the dense cube, two distances, subbins
        dict(name="dense-plan", form="plan", data="dense", traj=20000, samples=101, qtraj=500,
             kind="spatiotemporal", d="0.5,2", queries="device", rows="sorted"),
        # the largest: 20,000,000 segments, 400,000 query segments at two distances, about a
        # thousand million rows (the benchmark's default workload on one index)
        dict(name="merger-plan", form="plan", data="merger", traj=100000, samples=201, qtraj=2000,
             kind="spatial", d="1,5", queries="device", rows="device"),
        # the same database at a small distance, where the filters are most of the work
        dict(name="merger-near-plan", form="plan", data="merger", traj=100000, samples=201,
             qtraj=500, kind="temporal", d="1", queries="device", rows="sorted"),
        # twelve clients' requests of mixed sizes and distances through the request loop
        dict(name="merger-served", form="served", data="merger", traj=10000, samples=201, qtraj=200,
             requests=12, kind="spatial", d="0.5,5", queries="host", rows="device"),
        # all pairs without any allocation by the library
        dict(name="all-pairs", form="noalloc", data="walk", traj=500, samples=401, box=1000.0,
             sigma=2.0, spread=100.0, qtraj=25, kind="brute", d="10", queries="device",
             rows="sorted"),
        # a new database: build its index, then search it once
        dict(name="build-index", form="build", data="walk", traj=2500, samples=401, box=1000.0,
             sigma=2.0, spread=100.0, qtraj=5, kind="spatiotemporal", d="10", queries="device",
             rows="sorted"),
    ]


def draw(rng):
    def logi(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def logd(lo, hi):
        return float("%.3g" % math.exp(rng.uniform(math.log(lo), math.log(hi))))

    form = rng.choice(["search", "search", "points", "plan", "plan", "served", "noalloc", "build"])
    data = rng.choice(["walk", "dense", "merger"])
    if form in ("points", "noalloc"):
        data = "walk"
    kind = rng.choice(["spatial", "temporal", "spatiotemporal"])
    c = dict(form=form, data=data)
    if data == "walk":
        c.update(traj=logi(100, 2500), samples=logi(21, 401), box=1000.0, sigma=2.0,
                 spread=100.0)
        dist = (1.0, 25.0)
    elif data == "dense":
        c.update(traj=logi(1000, 20000), samples=rng.randint(51, 101))
        dist = (0.5, 2.0)
    else:
        c.update(traj=2 * logi(500, 50000), samples=rng.randint(101, 201))
        dist = (1.0, 5.0)
    ds = [logd(*dist) for _ in range(rng.randint(1, 3) if form == "plan" else 1)]
    if form == "points":
        q = logi(10, 2000)
    elif form == "noalloc":
        q = logi(2, 25)
        c["traj"] = min(c["traj"], 500)
        kind = "brute"
    elif form == "build":
        q = logi(1, 10)
    elif form == "served":
        q = logi(20, 100)
        c["requests"] = rng.randint(3, 12)
        kind = "spatial"
        ds = [dist[0], dist[1]]
    else:
        q = logi(1, max(2, c["traj"] // 50))
    c.update(qtraj=q, kind=kind, d=",".join("%g" % x for x in ds),
             queries="host" if form == "served" else rng.choice(["device", "host"])
             if form == "search" else "device",
             rows="device" if kind == "spatial" and form in ("search", "points", "plan",
                                                                      "served") else "sorted")
    return c


# ---------------------------------------------------------------------------------------------
# trajectories, drawn on the GPU
# ---------------------------------------------------------------------------------------------
def _uniform(gen, shape, lo, hi):
    return lo + (hi - lo) * torch.rand(shape, generator=gen, dtype=torch.float64, device=DEV)


def _normal(gen, shape, sigma):
    return sigma * torch.randn(shape, generator=gen, dtype=torch.float64, device=DEV)


def _columns(pos, t):
    """Segments of the trajectories: pos (traj, samples, 3), t (traj, samples); eight columns."""
    a, b = pos[:, :-1].reshape(-1, 3), pos[:, 1:].reshape(-1, 3)
    return tuple(x.contiguous() for x in (a[:, 0], a[:, 1], a[:, 2], t[:, :-1].reshape(-1),
                                          b[:, 0], b[:, 1], b[:, 2], t[:, 1:].reshape(-1)))


def _plummer(gen, n, a, rmax):
    """Radii of a Plummer sphere of scale a, cut at rmax (inverse of the cumulative mass)."""
    top = (1.0 + (a / rmax) ** 2) ** -1.5
    x = _uniform(gen, (n,), 0.0, top).clamp_min(1e-12)
    return a / torch.sqrt(x.pow(-2.0 / 3.0) - 1.0)


def _database(case, gen):
    """Columns of the database and the trajectories that queries are drawn from."""
    nt, ns = case["traj"], case["samples"]
    steps_t = torch.arange(ns, dtype=torch.float64, device=DEV)
    if case["data"] == "walk":
        p0 = _uniform(gen, (nt, 1, 3), 0.0, case["box"])
        steps = _normal(gen, (nt, ns - 1, 3), case["sigma"])
        t = _uniform(gen, (nt, 1), 0.0, case["spread"]) + steps_t
        pool = torch.arange(nt, device=DEV)
    elif case["data"] == "dense":
        p0 = _uniform(gen, (nt, 1, 3), 0.0, 50.0)
        steps = _normal(gen, (nt, ns - 1, 3), 0.5)
        t = steps_t.expand(nt, ns)
        pool = torch.arange(nt, device=DEV)
    else:
        half = nt // 2
        r = _plummer(gen, nt, 10.0, 100.0)
        v = _normal(gen, (nt, 3), 1.0)
        first = (torch.arange(nt, device=DEV) < half)[:, None]
        centre = torch.where(first, torch.tensor([-100.0, -5.0, 0.0], dtype=torch.float64, device=DEV),
                             torch.tensor([100.0, 5.0, 0.0], dtype=torch.float64, device=DEV))
        bulk = torch.where(first, torch.tensor([0.5, 0.0, 0.0], dtype=torch.float64, device=DEV),
                           torch.tensor([-0.5, 0.0, 0.0], dtype=torch.float64, device=DEV))
        p0 = (centre + r[:, None] * v / v.norm(dim=1, keepdim=True))[:, None]
        steps = bulk[:, None] + _normal(gen, (nt, ns - 1, 3), 0.1)
        t = steps_t.expand(nt, ns)
        pool = torch.nonzero(r < 10.0).reshape(-1)
    pos = torch.cat([p0, p0 + torch.cumsum(steps, 1)], 1)
    if case["data"] == "dense":  # reflecting walls
        u = torch.remainder(pos, 100.0)
        pos = torch.where(u > 50.0, 100.0 - u, u)
    return _columns(pos, t), pool


def _take(cols, traj, seg_per):
    idx = (traj[:, None] * seg_per + torch.arange(seg_per, device=DEV)).reshape(-1)
    return tuple(c[idx].contiguous() for c in cols)


def _make(case, seed):
    """(database columns, query columns, t_start, t_end): all on the device."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) * 7919 + 1410)
    db, pool = _database(case, gen)
    if case["form"] == "points":
        q = tuple(_uniform(gen, (case["qtraj"],), 0.0, case["box"]) for _ in range(3))
    else:
        pick = torch.randperm(pool.numel(), generator=gen, device=DEV)[:case["qtraj"]]
        q = _take(db, pool[pick].sort().values, case["samples"] - 1)
    return gen, db, q, float(db[3].min()), float(db[7].max())


def _distances(case):
    return [float(x) for x in case["d"].split(",")]


def _served_sizes(case):
    """Trajectories and run lengths of the clients' requests: 1 to qtraj trajectories
    (log-uniform), each a run of 10 to 200 segments; d log-uniform between the case's two."""
    seg, n = case["samples"] - 1, case["requests"]
    rng = np.random.Generator(np.random.PCG64(1410))
    lo, hi = _distances(case)
    share = rng.permutation(n) / max(1, n - 1)
    k = np.maximum(1, np.rint(case["qtraj"] ** share)).astype(np.int64)
    d = lo * (hi / lo) ** (rng.permutation(n) / max(1, n - 1))
    return [(np.minimum(rng.integers(10, 201, x), seg), float(y)) for x, y in zip(k, d)]


def _served_requests(case, gen, db):
    """The requests as clients send them: host arrays, runs of random database trajectories."""
    seg = case["samples"] - 1
    host = [c.cpu().numpy().reshape(case["traj"], seg) for c in db]
    rng = np.random.Generator(np.random.PCG64(int(torch.randint(1 << 40, (1,), generator=gen,
                                                                device=DEV))))
    out = []
    for length, d in _served_sizes(case):
        rows = rng.integers(0, case["traj"], length.size)
        first = rng.integers(0, seg - length + 1)
        cols = [np.concatenate([h[r, f:f + n] for r, f, n in zip(rows, first, length)])
                for h in host]
        out.append((cols, d, float(cols[3].min()), float(cols[7].max())))
    return out


# ---------------------------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------------------------
class _Array:
    """Device rows of the library as an array that torch can view; keeps their owner alive."""

    def __init__(self, ptr, n, typestr, owner):
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": typestr, "data": (ptr, False),
                                         "version": 2}
        self.owner = owner


_NAMES = ("q_idx", "e_idx", "t_in", "t_out")
_STR = ("<i4", "<i4", "<f8", "<f8")
_TYPES = (torch.int32, torch.int32, torch.float64, torch.float64)


def _views(ptrs, n, owner):
    if n == 0:
        return [torch.empty(0, dtype=t, device=DEV) for t in _TYPES]
    return [torch.as_tensor(_Array(p, n, t, owner), device=DEV) for p, t in zip(ptrs, _STR)]


def _row_room(case):
    """Rows that the program has room for, by request: half as many again as it expects, and more
    where few trajectories stand for the average."""
    seg = case["samples"] - 1
    if case["form"] == "served":
        want = [(n.sum(), n.size, d) for n, d in _served_sizes(case)]
    else:
        want = [(case["qtraj"] * seg, case["qtraj"], d) for d in _distances(case)]
    return [int((1.5 + 3.5 / math.sqrt(k)) * n * _rows_per_query(case, d)) + 4096
            for n, k, d in want]


def _buffers(case):
    """The program's own row arrays: a result's rows are handed on in them."""
    dev = "cpu" if case["rows"] == "sorted" and case["queries"] == "host" else DEV
    return [[torch.zeros(n, dtype=t, device=dev) for t in _TYPES] for n in _row_room(case)]


def _hand_on(case, rows, out, n, spans=(), nq=0):
    """The rows in the program's arrays, in (query, entry) order where it needs one; spans: (first,
    count) of the requests of one run, whose rows stay one request after another."""
    m = rows[0].numel()
    if case["rows"] == "sorted":
        key = torch.add(rows[1], rows[0].long(), alpha=n)
        for r, (a, c) in enumerate(spans):
            if r:
                key[a:a + c] += r * nq * n
        order = torch.argsort(key)
        for x, y in zip(rows, out):
            torch.index_select(x, 0, order, out=y[:m])
    else:
        for x, y in zip(rows, out):
            y[:m].copy_(x)
    return out


def _result(case, res, out, n):
    if case["rows"] == "sorted" and case["queries"] == "host":
        r = res.to_host(sort=True)
        for k, y in zip(_NAMES, out):
            y.numpy()[:res.count] = r[k]
        return out
    return _hand_on(case, _views(res.device_arrays() if res.count else (), res.count, res), out, n)


def prepare(case, seed):
    gen, db, q, t0, t1 = _make(case, seed)
    s = {"case": case, "n": db[0].numel(), "t": (t0, t1), "d": _distances(case)}
    form = case["form"]
    if form == "plan" and case["rows"] == "sorted":
        s["out"] = [torch.zeros(sum(_row_room(case)), dtype=t, device=DEV) for t in _TYPES]
    elif form != "plan":
        s["out"] = _buffers(case)
    if form == "noalloc":
        s.update(db=db, q=q, room=[torch.empty(_row_room(case)[0], dtype=t, device=DEV)
                                   for t in _TYPES])
        return s
    if form == "build":
        s.update(db=db, q=q)
        return s
    s["index"] = ix = api.ts_build_index(db, kind=case["kind"])
    if form == "served":
        s["requests"] = _served_requests(case, gen, db)
        s["server"] = api.Server(ix, max_batch_requests=16, max_batch_queries=1 << 18,
                                 max_batch_rows=1 << 25, mem_budget_bytes=16 << 30)
        return s
    if form == "plan":
        # the plan's capacities: tiles from searches that keep no rows, candidate ranges from the
        # schedule, rows as expected
        tiles = units = 0
        for d in s["d"]:
            r = api.ts_search(ix, q, d, t0, t1, max_results=1)
            tiles += r.stats["n_tiles"]
            r.free()
            if case["kind"] == "spatial":
                units += int(api.ts_schedule(ix, q, d, t0, t1)[1].sum())
        nq, rows = q[0].numel(), sum(_row_room(case))
        if case["queries"] == "pinned":
            q = tuple(c.cpu().pin_memory() for c in q)
        s["plan"] = api.BatchPlan(ix, max_requests=len(s["d"]), max_queries=nq * len(s["d"]),
                                  max_rows=rows, max_units=units,
                                  max_tiles=tiles + tiles // 4 + 65536, use_graph=True)
        s["requests"] = api.prepare_requests([(q, d, t0, t1) for d in s["d"]])
        s.update(rows=rows, nq=nq)
        if case["rows"] == "host":
            s["host"] = {k: torch.zeros(rows, dtype=t).pin_memory().numpy()
                         for k, t in zip(_NAMES, _TYPES)}
        return s
    s["q"] = [c.cpu().numpy() for c in q] if case["queries"] == "host" else q
    return s


def run(s):
    case, (t0, t1) = s["case"], s["t"]
    form = case["form"]
    if form == "search":
        res = api.ts_search(s["index"], s["q"], s["d"][0], t0, t1)
        return _result(case, res, s["out"][0], s["n"])
    if form == "points":
        res = api.ts_search_points(s["index"], *s["q"], s["d"][0], t0, t1)
        return _result(case, res, s["out"][0], s["n"])
    if form == "build":
        ix = api.ts_build_index(s["db"], kind=case["kind"])
        res = api.ts_search(ix, s["q"], s["d"][0], t0, t1)
        return [api.ts_index_export(ix, "perm").view(np.int32)] + _result(case, res, s["out"][0],
                                                                          s["n"])
    if form == "noalloc":
        st, n = api.ts_search_brute_noalloc(s["db"], s["q"], s["d"][0], t0, t1, *s["room"])
        if st:
            raise RuntimeError("more rows than the output arrays hold")
        return _hand_on(case, [x[:n] for x in s["room"]], s["out"][0], s["n"])
    if form == "served":
        srv = s["server"]
        tickets = [srv.submit(q, d, a, b) for q, d, a, b in s["requests"]]
        results = [srv.wait(t)[0] for t in tickets]
        return [_result(case, r, out, s["n"]) for r, out in zip(results, s["out"])]
    plan = s["plan"]
    plan.run(s["requests"])
    st = plan.wait()
    if st["overflow"]:
        raise RuntimeError("the plan's capacities were exceeded")
    if case["rows"] == "host":  # the first rows of the arrays, and each request's count
        rows, spans = plan.rows_to_host(out=s["host"])
        return [s["host"][k] for k in _NAMES] + [n for _, n in spans]
    ptrs = [ctypes.c_void_p() for _ in range(4)]
    _lib.check(_lib.load().ts_batch_rows(plan.handle, *[ctypes.byref(p) for p in ptrs]))
    rows = _views([p.value for p in ptrs], s["rows"], plan)  # the plan's own arrays, whole
    spans = [plan.request_rows(r) for r in range(len(s["d"]))]
    if case["rows"] == "sorted":
        rows = _hand_on(case, [x[:st["rows"]] for x in rows], s["out"], s["n"], spans, s["nq"])
    return rows + [n for _, n in spans]


# ---------------------------------------------------------------------------------------------
# the work of a pass, and its values in 64 bits
# ---------------------------------------------------------------------------------------------
def _rows_per_query(case, d):
    """About how many rows a query segment has: the entries alive with it, times the part of the
    space within d of it (two entries of a trajectory meet a segment whose times are not aligned)."""
    ball = 4.0 / 3.0 * math.pi * d ** 3
    if case["form"] == "points":  # (by a trajectory's segment: any of them may pass the point)
        return case["traj"] * min(1.0, ball / case["box"] ** 3)
    if case["data"] == "walk":
        span = case["samples"] - 1
        alive = case["traj"] * span / (span + case.get("spread", 0.0))
        return 1.0 + 2.0 * alive * min(1.0, ball / case["box"] ** 3)
    if case["data"] == "dense":
        return 1.0 + case["traj"] * ball / 50.0 ** 3
    return 1.0 + 0.4 * case["traj"] / 2 * min(1.0, ball * 3.0 / (4.0 * math.pi * 1000.0))


def work(case):
    """Each query read once (64 B), each entry's exact record once for each request (64 B), each row
    written once (24 B); per row the pair test in 64 bits (51 operations)."""
    n = case["traj"] * (case["samples"] - 1)
    ds = _distances(case)
    seg = case["samples"] - 1
    if case["form"] == "served":
        sizes = [(float(x.sum()), d) for x, d in _served_sizes(case)]
        nq, rows = sum(x for x, _ in sizes), sum(x * _rows_per_query(case, d) for x, d in sizes)
        return {"bytes": 64.0 * nq + 64.0 * n + 24.0 * rows, "flops": 51.0 * rows}
    if case["form"] == "points":
        nq = case["qtraj"]
        rows = nq * seg * _rows_per_query(case, ds[0])
        return {"bytes": 24.0 * nq + 64.0 * n + 24.0 * rows, "flops": 51.0 * rows}
    nq = case["qtraj"] * seg
    rows = sum(nq * _rows_per_query(case, d) for d in ds)
    # the entries that can meet some query: a query trajectory meets those near its path, at most
    # all of them (a search of few queries need not read the whole database)
    near = min(float(n), rows) if case["form"] != "noalloc" else float(n)
    out = {"bytes": 64.0 * nq + 64.0 * near + 24.0 * rows, "flops": 51.0 * rows}
    if case["form"] == "build":
        out["bytes"] += 64.0 * n + 4.0 * n + 96.0 * n  # columns in, order and exact records out
    return out


def _interval(q, e, d, ts, te):
    """Hit and interval of pairs (columns of equal length) in 64 bits: the common window of the two
    segments and [ts, te], and where on it the squared distance is at most d^2."""
    lo = torch.maximum(torch.maximum(q[3], e[3]), torch.full_like(q[3], ts))
    hi = torch.minimum(torch.minimum(q[7], e[7]), torch.full_like(q[3], te))
    r, v = [], []
    for k in range(3):
        qv, ev = (q[4 + k] - q[k]) / (q[7] - q[3]), (e[4 + k] - e[k]) / (e[7] - e[3])
        r.append((q[k] + qv * (lo - q[3])) - (e[k] + ev * (lo - e[3])))
        v.append(qv - ev)
    a = sum(x * x for x in v)
    b = sum(x * y for x, y in zip(r, v))
    c = sum(x * x for x in r) - d * d
    span = hi - lo
    disc = b * b - a * c
    s = -(b + torch.copysign(torch.sqrt(disc.clamp_min(0.0)), b))
    r1, r2 = s / a, c / s
    still = a == 0
    first = torch.where(still, torch.zeros_like(a), torch.minimum(r1, r2)).nan_to_num(0.0).clamp_min(0.0)
    last = torch.minimum(torch.where(still, span, torch.maximum(r1, r2).nan_to_num(0.0)), span)
    hit = (hi > lo) & torch.where(still, c <= 0, (disc >= 0) & (first <= last))
    return hit, lo + first, lo + last


def _exact_rows(db, q, d, ts, te, alive):
    """Every row in (query, entry) order, in 64 bits: pairs whose times and boxes meet, then the
    closed form."""
    n = db[0].numel()
    order = torch.argsort(db[3], stable=True)
    dbs = [c[order] for c in db]
    dur = float((db[7] - db[3]).max())
    emin = [torch.minimum(dbs[k], dbs[4 + k]) for k in range(3)]
    emax = [torch.maximum(dbs[k], dbs[4 + k]) for k in range(3)]
    qorder = torch.argsort(q[3], stable=True)
    keys, tins, touts = [], [], []
    step = max(1, min(4096, (1 << 26) // int(1 + min(alive, 1 << 20))))
    for f in range(0, q[0].numel(), step):
        sel = qorder[f:f + step]
        qq = [c[sel] for c in q]
        a = int(torch.searchsorted(dbs[3], max(float(qq[3].min()), ts) - dur * 1.001 - 1e-6))
        b = int(torch.searchsorted(dbs[3], min(float(qq[7].max()), te)))
        for lo in range(a, b, 1 << 20):
            part = slice(lo, min(b, lo + (1 << 20)))
            near = (dbs[3][part] < qq[7][:, None]) & (dbs[7][part] > qq[3][:, None])
            for k in range(3):
                qlo, qhi = torch.minimum(qq[k], qq[4 + k]) - d, torch.maximum(qq[k], qq[4 + k]) + d
                near &= (emax[k][part] >= (qlo - 1e-6)[:, None]) & (emin[k][part] <= (qhi + 1e-6)[:, None])
            i, j = torch.nonzero(near, as_tuple=True)
            j = j + lo
            hit, tin, tout = _interval([c[i] for c in qq], [c[j] for c in dbs], d, ts, te)
            keys.append((sel[i] * n + order[j])[hit])
            tins.append(tin[hit])
            touts.append(tout[hit])
    key = torch.cat(keys) if keys else torch.empty(0, dtype=torch.int64, device=DEV)
    at = torch.argsort(key)
    return [None, None] + [torch.cat(x)[at] if x else torch.empty(0, dtype=torch.float64, device=DEV)
                           for x in (tins, touts)]


def exact(case, seed):
    # rows that come in the library's own order have no value that only the inputs give
    if case["rows"] != "sorted":
        return None
    gen, db, q, t0, t1 = _make(case, seed)
    n, nq = db[0].numel(), q[0].numel()
    alive = n if case["form"] in ("points", "noalloc") else 3.0 * n / max(1, case["samples"] - 1)
    if nq * len(_distances(case)) * alive > 6e10:  # about 20 seconds
        return None
    if case["form"] == "points":
        q = (*q, torch.full((nq,), t0, dtype=torch.float64, device=DEV), *q,
             torch.full((nq,), t1, dtype=torch.float64, device=DEV))
    rows = [_exact_rows(db, q, d, t0, t1, alive) for d in _distances(case)]
    if case["form"] == "plan":  # its requests' rows one after another
        rows = [[None, None] + [torch.cat([r[k] for r in rows]) for k in (2, 3)]]
    room = sum(_row_room(case))
    rows = [None, None] + [torch.cat([rows[0][k], torch.zeros(room - rows[0][k].numel(),
                                                              dtype=torch.float64, device=DEV)])
                           for k in (2, 3)]
    return [None] + rows if case["form"] == "build" else rows

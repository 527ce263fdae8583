"""The calls a user of the minimiser makes, over the range of sizes and options
in use, for timing them and for comparing their results.

Every case goes through the package's public entry points: ``Solver.solve``
(whole branch-and-bound solves, plain and in the paper's own procedure),
``Solver.eval_boxes`` (interval values and partials of given boxes),
``Solver.resume`` / ``snapshot`` (checkpoint and resume of the region list) and
``Server`` (many problems at once).  A seed gives a problem's coefficients, its
planted minimiser and its boxes; the paper's functions have no coefficients,
there the seed moves the domain's bounds.

Solves carry a generation limit a little above what the seed-0 problem needs,
so a hard seed ends with the rigorous enclosure of a limited solve instead of
running on.
"""
import math
import time

import numpy as np
import torch

import paper_2507_01770_gb300 as gb
import synthetic as S

GIB = 1 << 30


# ---------------------------------------------------------------------------
# cases
def listed():
    return [
        # one box of a 2-variable objective: what one call costs before any work
        dict(name="eval_one_box", kind="eval", family="sep_cos", n=2, block=2, nbox=1, blk=0, fp32=False),
        # re-evaluating a pool of boxes of the n = 100 chain with their partials, FP64
        dict(name="eval_chain100", kind="eval", family="chain", n=100, block=10, nbox=8192, blk=5, fp32=False),
        # a few hundred boxes of the largest objective in FP32, odd sizes, the
        # last cycling block holding a single coordinate
        dict(name="eval_mixed10001_f32", kind="eval", family="mixed", n=10001, block=100, nbox=301, blk=100, fp32=True),
        # the 2-variable problem at width 1e-8 with the default options
        dict(name="solve_n2", kind="solve", family="sep_cos", n=2, block=2, tol=1e-8, split_m=2, split_d=0,
             max_children=1 << 22, fp32=0, sync=0, max_gens=200, pool_gib=2, device_only=False),
        # several parents per generation, FP32 prefilter, ragged last block
        dict(name="solve_chain23_batched", kind="solve", family="chain", n=23, block=10, tol=1e-6, split_m=2,
             split_d=5, max_children=16 * 32, fp32=1, sync=4, max_gens=400, pool_gib=2, device_only=False),
        # the n = 100 chain in FP64: 4^10 children of one box per generation
        dict(name="solve_chain100", kind="solve", family="chain", n=100, block=10, tol=1e-6, split_m=4, split_d=10,
             max_children=1 << 20, fp32=0, sync=0, max_gens=160, pool_gib=8, device_only=False),
        # the n = 1000 exp/sqrt/cos family, 2^10 children, FP32 then FP64, graph replays
        dict(name="solve_ackley1000", kind="solve", family="ackley", n=1000, block=10, tol=1e-6, split_m=2, split_d=10,
             max_children=1 << 10, fp32=1, sync=16, max_gens=3000, pool_gib=8, device_only=False),
        # the n = 10^4 mixed family, block-record pool, result left on the device
        dict(name="solve_mixed10000", kind="solve", family="mixed", n=10000, block=100, tol=1e-6, split_m=2,
             split_d=10, max_children=1 << 10, fp32=1, sync=16, max_gens=22500, pool_gib=24, device_only=True),
        # the paper's own procedure on its Levy function, n = 30: 4^10 children of one
        # region, 10 diagonal samples, every coordinate tested, regions to width 1e-4
        dict(name="paper_levy30", kind="paper", family="paper_levy", n=30, split_d=10, max_gens=27, pool_gib=8),
        # the same on a product form, the last block of 6 coordinates, stopped early
        dict(name="paper_griewank16", kind="paper", family="paper_griewank", n=16, split_d=10, max_gens=10, pool_gib=4),
        # sixteen requests of the serving stream at once (n log-uniform in 2 .. 600)
        dict(name="serve_16", kind="serve", count=16, n_max=600),
        # a stopped n = 100 solve taken up from its snapshot, run on and saved again
        dict(name="resume_chain100", kind="resume", n=100, block=10, split_m=4, split_d=6, parents=4, first=24, more=12),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "solve", "solve", "solve", "wide", "paper", "serve", "resume"])
    if kind == "eval":
        family = rng.choice(["sep_cos", "chain", "ackley", "mixed"])
        n = _log_int(rng, 2, 10000)
        block = min(n, 100 if family == "mixed" and n >= 200 else 10)
        nbox = _log_int(rng, 1, min(65536, max(2, (1 << 22) // n)))
        nb = (n + block - 1) // block
        return dict(kind="eval", family=family, n=n, block=block, nbox=nbox,
                    blk=rng.choice([-1, 0, nb - 1, rng.randrange(nb)]), fp32=rng.random() < 0.5)
    if kind == "solve":   # one best box per generation (the serving setting), or a few
        family = rng.choice(["sep_cos", "chain", "ackley", "mixed"])
        n = _log_int(rng, 128 if family == "mixed" else 2, 8000 if family == "mixed" else 2000)
        block = min(n, 100 if family == "mixed" else 10)
        d = rng.choice([min(block, 10), (min(block, 10) + 1) // 2])
        parents = rng.choice([1, 1, 1, 4])
        return dict(kind="solve", family=family, n=n, block=block, tol=1e-6, split_m=2, split_d=d,
                    max_children=parents << d, fp32=int(rng.random() < 0.7), sync=rng.choice([0, 4, 16]),
                    max_gens=rng.randrange(200, 1200), pool_gib=4, device_only=n > 64)
    if kind == "wide":    # a large fan-out of one box per generation, FP64
        family = rng.choice(["sep_cos", "chain", "ackley"])
        n = _log_int(rng, 10, 200)
        return dict(kind="solve", family=family, n=n, block=10, tol=1e-6, split_m=4, split_d=rng.randrange(7, 11),
                    max_children=1 << 20, fp32=rng.randrange(2), sync=0, max_gens=rng.randrange(8, 40), pool_gib=8,
                    device_only=n > 30)
    if kind == "paper":
        return dict(kind="paper", family=rng.choice(["paper_levy", "paper_rastrigin", "paper_ackley", "paper_griewank"]),
                    n=rng.randrange(10, 51), split_d=rng.randrange(7, 11), max_gens=rng.randrange(4, 9), pool_gib=4)
    if kind == "serve":
        return dict(kind="serve", count=rng.randrange(2, 17), n_max=_log_int(rng, 20, 600))
    return dict(kind="resume", n=_log_int(rng, 12, 120), block=10, split_m=rng.choice([2, 4]), split_d=5,
                parents=rng.choice([1, 2, 4]), first=rng.randrange(8, 24), more=rng.randrange(4, 16))


# ---------------------------------------------------------------------------
# what a user's program has in hand
def _problem(case, seed):
    return S.make(case["family"], n=case["n"], seed=seed, block=case["block"], **({"tol_f": case["tol"]} if "tol" in case else {}))


def _boxes(case, seed):
    p = _problem(case, seed)
    return p, *S.random_boxes(p, case["nbox"], seed=seed + 1, around_s=0.3)


def _chain_solver(case, p, gens):
    fan = case["split_m"] ** case["split_d"]
    return gb.Solver(p, block=case["block"], split_m=case["split_m"], split_d=case["split_d"],
                     max_children=case["parents"] * fan, max_generations=gens, pool_mode=1, gens_per_sync=4,
                     pool_bytes=4 * GIB)


def _rows(n):
    """Room of the caller's for region bounds (4M numbers)."""
    return np.full(((1 << 22) // n, n), np.nan)


def _regions(n, gens):
    """The caller's arrays that a result's regions and per-generation rows go to."""
    return dict(box_lo=_rows(n), box_hi=_rows(n), box_flo=np.full((1 << 22) // n, np.nan),
                trace=np.zeros((5, gens), dtype=np.int64), gub=np.zeros(gens))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "eval":
        p, lo, hi = _boxes(case, seed)
        return dict(kind=kind, solver=gb.Solver(p, block=case["block"], pool_bytes=64 << 20), blk=case["blk"],
                    fp32=case["fp32"], lo=torch.from_numpy(lo).cuda(), hi=torch.from_numpy(hi).cuda())
    if kind == "solve":
        p = _problem(case, seed)
        return dict(kind=kind, device_only=case["device_only"], **_regions(case["n"], case["max_gens"]),
                    solver=gb.Solver(p, block=case["block"], split_m=case["split_m"], split_d=case["split_d"],
                                     max_children=case["max_children"], fp32_prefilter=case["fp32"],
                                     gens_per_sync=case["sync"], max_generations=case["max_gens"],
                                     pool_bytes=case["pool_gib"] * GIB))
    if kind == "paper":
        p = S.make(case["family"], n=case["n"])
        r = np.random.Generator(np.random.PCG64(seed))
        w = p.u - p.l
        p.l = p.l - w * r.uniform(0.0, 0.02, p.n)
        p.u = p.u + w * r.uniform(0.0, 0.02, p.n)
        return dict(kind=kind, device_only=False, **_regions(case["n"], case["max_gens"]),
                    solver=gb.Solver(p, block=10, split_m=4, split_d=case["split_d"],
                                     max_children=4 ** case["split_d"], samples=10, mono_all=1, tol_x=1e-4,
                                     max_generations=case["max_gens"], pool_bytes=case["pool_gib"] * GIB))
    if kind == "serve":
        stream = [p for _, p in S.serving_stream(count=case["count"], seed=seed, n_max=case["n_max"])]
        opts = [gb.gb_default_options(block=min(p.n, 10), split_m=2, split_d=min(p.n, 10), max_children=1 << 10,
                                      fp32_prefilter=1, pool_bytes=4 * GIB, gens_per_sync=4, max_generations=4000)
                for p in stream]
        return dict(kind=kind, server=gb.Server(case["count"] * 4 * GIB, max_active=16), stream=stream, opts=opts,
                    **_regions(1, 1))
    p = S.chain(n=case["n"], seed=seed, block=case["block"])
    s = _chain_solver(case, p, case["first"])
    s.solve(device_only=True, raise_on_error=False)
    snap = s.snapshot()
    s.close()
    return dict(kind=kind, solver=_chain_solver(case, p, case["more"]), snap=snap,
                **_regions(case["n"], case["more"]), snap_lo=_rows(case["n"]), snap_hi=_rows(case["n"]),
                snap_flo=_rows(case["n"])[:, 0].copy(), snap_cyc=np.zeros(len(_rows(case["n"])), dtype=np.int32))


# ---------------------------------------------------------------------------
# one pass
def _keep(buf, rows):
    """rows into the caller's array (what does not fit is left)."""
    if rows is not None:
        k = min(len(buf), len(rows))
        buf[:k] = rows[:k]
    return buf


def _result(state, r):
    for i, k in enumerate(("parents", "children", "kept32", "kept", "pool")):
        _keep(state["trace"][i], r.trace[k])
    return dict(enclosure=np.array([r.fmin_lo, r.fmin_hi]),
                counts=np.array([r.status, r.n_boxes, r.generations, r.box_evals_fp32, r.box_evals_fp64, r.mid_evals]),
                trace=state["trace"], gub=_keep(state["gub"], r.trace["gub"]), box_lo=_keep(state["box_lo"], r.box_lo),
                box_hi=_keep(state["box_hi"], r.box_hi), box_flo=_keep(state["box_flo"], r.box_flo))


def run(state):
    kind = state["kind"]
    if kind == "eval":
        F, Fmid, G, mono = state["solver"].eval_boxes(state["lo"], state["hi"], state["blk"], state["fp32"])
        return dict(F=F, Fmid=Fmid, G=G, mono=mono)
    if kind in ("solve", "paper"):
        return _result(state, state["solver"].solve(device_only=state["device_only"], raise_on_error=False))
    if kind == "resume":
        out = _result(state, state["solver"].resume(state["snap"], raise_on_error=False))
        s = state["solver"].snapshot()
        out.update(snap_lo=_keep(state["snap_lo"], s.lo), snap_hi=_keep(state["snap_hi"], s.hi),
                   snap_flo=_keep(state["snap_flo"], s.flo), snap_cyc=_keep(state["snap_cyc"], s.cyc),
                   snap_gub=float(s.gub), snap_generations=int(s.generations))
        return out
    server = state["server"]
    ids = [server.submit(p, o) for p, o in zip(state["stream"], state["opts"])]
    done = {}
    while len(done) < len(ids):
        for i in ids:
            if i not in done:
                r = server.poll(i)
                if r is not None:
                    done[i] = r
        if len(done) < len(ids):
            time.sleep(0.0002)
    rs = [done[i] for i in ids]
    flat = lambda k: np.concatenate([getattr(r, k).reshape(-1, 1) for r in rs if getattr(r, k) is not None])  # noqa: E731
    return dict(enclosure=np.array([[r.fmin_lo, r.fmin_hi] for r in rs]),
                counts=np.array([[r.status, r.n_boxes, r.generations, r.box_evals_fp32, r.box_evals_fp64] for r in rs]),
                box_lo=_keep(state["box_lo"], flat("box_lo")), box_hi=_keep(state["box_hi"], flat("box_hi")),
                box_flo=_keep(state["box_flo"][:, None], flat("box_flo")))


# ---------------------------------------------------------------------------
# the work a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind == "eval":   # bounds in, results out; about 12 directed operations per term for F, 6 for the midpoint
        n, k = case["n"], case["nbox"]
        g = min(case["block"], n) if case["blk"] >= 0 else 0
        return {"bytes": k * (16.0 * n + 36.0 + 16.0 * g), "flops": k * (18.0 * n + 24.0 * g)}
    if kind == "serve":  # per request some hundreds of generations of 2^10 children
        kids = case["count"] * 300 * 1024.0
        return {"bytes": kids * 8.0, "flops": kids * 8.0}
    if kind == "resume":
        kids = case["more"] * case["parents"] * float(case["split_m"] ** case["split_d"])
        return {"bytes": kids * 8.0 + 16.0 * case["n"] * 4096, "flops": kids * 8.0}
    if kind == "paper":  # per child at least one addition for F and for each of the 10 samples
        kids = case["max_gens"] * 4.0 ** case["split_d"]
        return {"bytes": kids * 8.0, "flops": kids * 24.0}
    fan = case["split_m"] ** (case["split_d"] or min(case["block"], 10))
    gens = case["max_gens"] if case["n"] > 2 else 30
    kids = gens * float(fan if case["n"] > 2 else 1 << 10)
    # per child a value and a sample from its parent's (two additions each), its bound written
    return {"bytes": kids * 8.0 + 16.0 * case["n"], "flops": kids * 8.0}


# ---------------------------------------------------------------------------
# 64-bit values of the evaluation cases, by plain interval arithmetic in numpy
def _mul(x, y):
    with np.errstate(invalid="ignore"):
        p = [a * b for a in x for b in y]
    p = [np.where(np.isnan(v), 0.0, v) for v in p]   # 0 * inf = 0
    return np.minimum(np.minimum(p[0], p[1]), np.minimum(p[2], p[3])), np.maximum(np.maximum(p[0], p[1]), np.maximum(p[2], p[3]))


def _add(x, y):
    return x[0] + y[0], x[1] + y[1]


def _neg(x):
    return -x[1], -x[0]


def _sub(x, y):
    return _add(x, _neg(y))


def _sqr(x):
    a, b = x[0] * x[0], x[1] * x[1]
    return np.where((x[0] <= 0) & (x[1] >= 0), 0.0, np.minimum(a, b)), np.maximum(a, b)


def _cos(x):
    a, b = np.cos(x[0]), np.cos(x[1])
    lo, hi = np.minimum(a, b), np.maximum(a, b)
    k0, k1 = np.ceil(x[0] / np.pi), np.floor(x[1] / np.pi)
    has = k0 <= k1
    two, even = k0 + 1 <= k1, np.mod(k0, 2) == 0
    hi = np.where(has & (even | two), 1.0, hi)
    lo = np.where(has & (~even | two), -1.0, lo)
    wide = x[1] - x[0] >= 2 * np.pi
    return np.where(wide, -1.0, lo), np.where(wide, 1.0, hi)


def _sin(x):
    return _cos((x[0] - np.pi / 2, x[1] - np.pi / 2))


def _pt(v):
    return v, v


def _rcp(y):
    ok = (y[0] > 0) | (y[1] < 0)
    with np.errstate(divide="ignore"):
        return np.where(ok, 1.0 / y[1], -np.inf), np.where(ok, 1.0 / y[0], np.inf)


def _total(x):
    return x[0].sum(axis=1), x[1].sum(axis=1)


def _sep_value(a, b, y):
    return _add(_mul(_pt(a), _sqr(y)), _mul(_pt(b), _sub(_pt(1.0), _cos(_mul(_pt(2 * np.pi), y)))))


def _sep_slope(a, b, y):
    s = _sin(_mul(_pt(2 * np.pi), y))
    return _add(_mul(_pt(a), _mul(_pt(2.0), y)), _mul(_mul(_pt(b), s), _pt(2 * np.pi)))


def _chain_value(al, be, y0, y1):
    return _add(_mul(_pt(al), _sqr(_sub(y1, _sqr(y0)))), _mul(_pt(be), _sqr(y0)))


def _chain_slopes(al, be, y0, y1):
    """Adjoints of y0 and y1 in alpha (y1 - y0^2)^2 + beta y0^2."""
    d = _mul(_pt(al), _mul(_pt(2.0), _sub(y1, _sqr(y0))))
    two = _mul(_pt(2.0), y0)
    return _add(_mul(_neg(d), two), _mul(_pt(be), two)), d


def _cut(y, ix):
    return y[0][:, ix], y[1][:, ix]


def _exact_rows(p, y, block, blk):
    """F and, for blk >= 0, the partials of the block, of boxes with y = x - s."""
    n, t = p.n, p.tables
    c0, c1 = (blk * block, min(n, (blk + 1) * block)) if blk >= 0 else (0, 0)
    k = len(y[0])
    G = np.full((2, k, c1 - c0), 0.0)

    def put(ix, v):   # adds the adjoints v of coordinates ix to the block's partials
        m = (ix >= c0) & (ix < c1)
        if m.any():
            G[0][:, ix[m] - c0] += v[0][:, m]
            G[1][:, ix[m] - c0] += v[1][:, m]

    lo, hi = max(0, c0 - 1), c1
    if p.family == "sep_cos":
        F = _total(_sep_value(t[0], t[1], y))
        ix = np.arange(c0, c1)
        put(ix, _sep_slope(t[0][ix], t[1][ix], _cut(y, ix)))
    elif p.family in ("chain", "mixed"):
        if p.family == "chain":
            al, be, ci = t[0], t[1], np.arange(0, n - 1)
            F = _pt(np.zeros(k))
        else:
            al, be, ci = t[2], t[3], np.arange(1, n - 1, 2)
            ev = np.arange(0, n, 2)
            F = _total(_sep_value(t[0][ev], t[1][ev], _cut(y, ev)))
            e = ev[(ev >= c0) & (ev < c1)]
            put(e, _sep_slope(t[0][e], t[1][e], _cut(y, e)))
            if n % 2 == 0:   # the last odd coordinate has no successor
                last = np.array([n - 1])
                F = _add(F, _total(_mul(_pt(be[last]), _sqr(_cut(y, last)))))
                put(last, _mul(_pt(be[last]), _mul(_pt(2.0), _cut(y, last))))
        F = _add(F, _total(_chain_value(al[ci], be[ci], _cut(y, ci), _cut(y, ci + 1))))
        c = ci[(ci >= lo) & (ci < hi)]
        d0, d1 = _chain_slopes(al[c], be[c], _cut(y, c), _cut(y, c + 1))
        put(c, d0)
        put(c + 1, d1)
    else:                    # ackley
        g, two_pi = t[0], _pt(2 * np.pi)
        s1, s2, s3 = _total(_sqr(y)), _total(_cos(_mul(two_pi, y))), _total(_mul(_pt(g), _sqr(y)))
        q = np.sqrt(s1[0] / n), np.sqrt(s1[1] / n)
        ea = np.exp(-0.2 * q[1]), np.exp(-0.2 * q[0])
        ec = np.exp(s2[0] / n), np.exp(s2[1] / n)
        F = _add(_add(_mul(_pt(-20.0), ea), _neg(ec)), _add(_pt(20.0 + math.e), s3))
        a1 = _mul(_mul(_mul(_pt(-20.0), ea), _pt(-0.2)), _mul(_pt(0.5), _rcp(q)))
        a1, a2 = _mul(a1, _pt(1.0 / n)), _mul(_neg(ec), _pt(1.0 / n))
        ix = np.arange(c0, c1)
        yb = _cut(y, ix)
        col = lambda v: (v[0][:, None], v[1][:, None])  # noqa: E731
        if len(ix):
            put(ix, _mul(col(a1), _mul(_pt(2.0), yb)))
            put(ix, _mul(col(a2), _mul(_neg(_sin(_mul(two_pi, yb))), two_pi)))
            put(ix, _mul(_pt(g[ix]), _mul(_pt(2.0), yb)))
    return np.stack(F, axis=-1), np.stack([G[0], G[1]], axis=-1)


def exact(case, seed):
    if case["kind"] != "eval":
        return None          # the bounds of a search have no closed value
    p, lo, hi = _boxes(case, seed)
    s, block, blk = p.tables[{"sep_cos": 2, "chain": 2, "ackley": 1, "mixed": 4}[p.family]], case["block"], case["blk"]
    F, Fmid = np.empty((len(lo), 2)), np.empty((len(lo), 2))
    G = np.full((len(lo), block, 2), np.nan)
    step = max(1, (1 << 20) // p.n)
    for i in range(0, len(lo), step):
        y = lo[i:i + step] - s, hi[i:i + step] - s
        m = 0.5 * lo[i:i + step] + 0.5 * hi[i:i + step] - s
        F[i:i + step], g = _exact_rows(p, y, block, blk)
        Fmid[i:i + step] = _exact_rows(p, (m, m), block, -1)[0]
        if blk >= 0:
            G[i:i + step, :g.shape[1]] = g
    return dict(F=F, Fmid=Fmid, G=G, mono=None)

"""Where a generation changes from one plan to another: child counts on both
sides of what one block lists (8192) and of what several threads per child take
(16,384), pools on both sides of what one block selects from (16,384 entries,
many of them with equal keys), launched one by one and replayed, against the
oracle; child groups under graph replays, with idle parents and on block
records, against the walk over every child."""
import numpy as np
import pytest

import oracle as O
import synthetic as S
from synthetic.dag import Dag
from synthetic.families import Problem

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2507_01770_gb300 as gb  # noqa: E402

TRACE = ("parents", "children", "kept32", "kept", "pool", "gub")


def _double_well(n, B):
    # sum (x_i^2 - 1)^2: the boxes of a generation share a few lower bounds
    g = Dag()
    root = g.isum(g.sqr(g.sub(g.sqr(g.ivar(0)), g.const(1.0))), 0, n, 1)
    return Problem("double_well", n, g.nodes(), root, g.tables, np.full(n, -3.0), np.full(n, 3.0), 1e-6, B, np.ones(n), 0)


@pytest.mark.parametrize("sync", [0, 4])
@pytest.mark.parametrize("fam,n,B,d,K,gens", [
    ("chain", 12, 3, 3, 1024, 9), ("chain", 12, 3, 3, 1025, 9),     # 8192 and 8200 children
    ("chain", 12, 3, 3, 2048, 9), ("chain", 12, 3, 3, 2049, 9),     # 16,384 and 16,392
    ("chain", 18, 8, 3, 1100, 8), ("chain", 33, 16, 3, 1100, 12),   # 8 and 16 threads a child
    ("double_well", 12, 3, 3, 700, 13), ("double_well", 15, 3, 3, 1500, 14),
])
def test_small_fan_outs(fam, n, B, d, K, gens, sync):
    p = _double_well(n, B) if fam == "double_well" else S.chain(n=n, seed=4, block=B)
    s = gb.Solver(p, block=B, split_m=2, split_d=d, max_children=K << d, max_generations=gens, gens_per_sync=sync,
                  pool_bytes=1 << 30)
    g = s.solve(raise_on_error=False)
    s.close()
    o = O.Oracle(p, block=B).solve(tol_f=p.tol_f, split_m=2, split_d=d, max_parents=K, max_gen=gens, threads=8)
    for k in ("parents", "children", "kept", "pool", "gub"):
        assert np.array_equal(g.trace[k], o.trace[k]), k
    assert g.fmin_lo == o.glb and g.fmin_hi == o.gub
    assert np.array_equal(g.box_lo, o.box_lo) and np.array_equal(g.box_flo, o.box_flo)
    assert g.trace["children"].max() == K << d


@pytest.mark.parametrize("groups", [56, 57, 58])
def test_shared_memory_around_what_needs_no_asking(groups):
    # 8 threads a child, a kernel of groups * 512 + nodes * 32 bytes and 20 KB more: every step of
    # 32 bytes around the 48 KB that a launch gets, the kernel's own arrays included
    n = 8 * groups
    for nodes in range(17):
        g = Dag()
        t = g.sqr(g.ivar(0))
        for _ in range(nodes):
            t = g.neg(t)
        if nodes % 2:
            t = g.neg(t)
        root = g.isum(t, 0, n, 1)
        p = Problem("squares", n, g.nodes(), root, g.tables, np.full(n, -1.0), np.full(n, 2.0), 1e-6, 8,
                    np.zeros(n), 0)
        s = gb.Solver(p, block=8, split_m=2, split_d=3, max_children=8, max_generations=3, pool_bytes=1 << 26)
        r = s.solve(raise_on_error=False)
        s.close()
        assert r.status == gb.GB_E_LIMIT and r.generations == 3, (groups, nodes, r.status, gb.gb_last_error())


@pytest.mark.parametrize("sync", [0, 3])
@pytest.mark.parametrize("pool_mode", [1, 2])
@pytest.mark.parametrize("fam,mode,K,extra", [
    ("chain", 3, 1, {}), ("mixed", 3, 3, {}), ("paper_levy", 0, 1, dict(samples=5, mono_all=1, tol_x=1e-3)),
    ("paper_griewank", 0, 3, dict(samples=5, mono_all=1, tol_x=1e-3))])
def test_groups(fam, mode, K, extra, pool_mode, sync):
    p = S.make(fam, n=24, block=6, **({} if fam.startswith("paper") else {"seed": 5}))
    r = []
    for m, g in ((mode, sync), (1, 0)):
        s = gb.Solver(p, eval_mode=m, block=6, split_m=4, split_d=6, max_children=K << 12, max_generations=14, tol_f=1e-6,
                      pool_mode=pool_mode, pool_bytes=1 << 30, gens_per_sync=g, **extra)
        r.append(s.solve(raise_on_error=False))
        s.close()
    a, b = r
    assert a.status == b.status and a.fmin_lo == b.fmin_lo and a.fmin_hi == b.fmin_hi
    for k in TRACE:
        assert np.array_equal(a.trace[k], b.trace[k]), k
    assert np.array_equal(a.box_lo, b.box_lo) and np.array_equal(a.box_hi, b.box_hi)
    assert np.array_equal(a.box_flo, b.box_flo)
    assert (a.box_evals_fp64, a.mid_evals) == (b.box_evals_fp64, b.mid_evals)
    assert a.ops64 < b.ops64   # (the work counted in the kernels: the tables were used)


@pytest.mark.parametrize("terms", [0, 1, 2])
@pytest.mark.parametrize("fp32", [False, True])
def test_boxes_of_objectives_with_hardly_a_term(terms, fp32):
    # no sum, sums of one term (one thread a box) and of two (several)
    n = 3
    g = Dag()
    root = g.mul(g.sqr(g.sub(g.var(0), g.const(0.25))), g.var(2))
    for off in (0, 1):
        if terms:
            t = g.sqr(g.sub(g.ivar(off), g.const(0.5)))
            root = g.add(root, g.isum(t, 0, terms, 1))
    p = Problem("few_terms", n, g.nodes(), root, g.tables, np.full(n, -2.0), np.full(n, 3.0), 1e-6, 2, np.zeros(n), 0)
    s = gb.Solver(p, block=2, pool_bytes=1 << 26)
    orc = O.Oracle(p, block=2)
    lo, hi = S.random_boxes(p, 150, seed=3)
    dlo, dhi = torch.from_numpy(lo).cuda(), torch.from_numpy(hi).cuda()
    for blk in (0, 1):
        w = min(2, n - 2 * blk)
        for noalloc in (False, True):
            F, Fm, G, mono = (t.cpu().numpy() for t in gb.gb_eval_boxes(s.h, dlo, dhi, blk, fp32, noalloc=noalloc))
            for k in range(0, 150, 7):
                f, fm, gr, m = orc.eval_box(lo[k], hi[k], blk=blk, f32=fp32)
                assert np.array_equal(F[k], f) and np.array_equal(Fm[k], fm)
                assert np.array_equal(G[k, :w], np.asarray(gr)[:w]) and mono[k] == m
    s.close()

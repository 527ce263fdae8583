"""A snapshot taken up under another split: regions then wait at cycling
positions for which the problem has no table layout (the tables are laid out at
the positions its own split reaches).  No region may be lost: the resumed solve
is the interpreter's, generation by generation, from term tables and in paper
mode, launched one by one and replayed, and the problem's next solve from the
domain is what it was."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2507_01770_gb300 as gb  # noqa: E402


def _same(a, b):
    assert a.status == b.status and a.generations == b.generations
    for k in ("parents", "children", "kept32", "kept", "pool", "gub"):
        assert np.array_equal(a.trace[k], b.trace[k]), k
    assert a.fmin_lo == b.fmin_lo and a.fmin_hi == b.fmin_hi and a.n_boxes == b.n_boxes
    assert np.array_equal(a.box_lo, b.box_lo) and np.array_equal(a.box_hi, b.box_hi)
    assert np.array_equal(a.box_flo, b.box_flo)


def _positions(n, B, d):
    return {c for b in range(0, n, B) for c in range(b, min(n, b + B), d)}


PAPER = dict(samples=5, mono_all=1, tol_x=1e-3)


@pytest.mark.parametrize("sync", [0, 4])
@pytest.mark.parametrize("fam,mode,first,then", [
    # one child block of 32 for sums, for any outer expression; one child per thread; in groups
    ("chain", 0, dict(block=10, split_d=5), dict(block=10, split_d=10, fp32_prefilter=1)),
    ("ackley", 0, dict(block=10, split_d=5), dict(block=10, split_d=10)),
    ("chain", 3, dict(block=10, split_d=5), dict(block=10, split_d=10)),
    ("ackley", 3, dict(block=10, split_d=3), dict(block=10, split_d=6)),
    # paper mode: by tables, products included; another block size
    ("paper_levy", 0, dict(block=10, split_d=5, **PAPER), dict(block=10, split_d=10, **PAPER)),
    ("paper_griewank", 0, dict(block=10, split_d=5, **PAPER), dict(block=10, split_d=6, **PAPER)),
    ("paper_levy", 0, dict(block=6, split_d=6, **PAPER), dict(block=10, split_d=5, **PAPER)),
])
def test_no_region_is_lost(fam, mode, first, then, sync):
    n = 20
    p = S.make(fam, n=n, block=10, **({} if fam.startswith("paper") else {"seed": 3}))
    a = gb.Solver(p, split_m=2, max_children=4 << first["split_d"], max_generations=7, tol_f=1e-6, **first)
    a.solve(raise_on_error=False)
    snap = a.snapshot()
    a.close()
    at = set((snap.cyc & 0x7fffffff).tolist())
    assert at - _positions(n, then["block"], then["split_d"]), "every region waits where the tables have a layout"
    opts = dict(split_m=2, max_children=2 << then["split_d"], max_generations=12, tol_f=1e-6, pool_mode=1,
                gens_per_sync=sync, **then)
    r = []
    for m in (mode, 1):
        s = gb.Solver(p, eval_mode=m, **opts)
        before = s.solve(raise_on_error=False) if sync else None   # (graphs of the tables are captured)
        r.append(s.resume(snap, raise_on_error=False))
        after = s.solve(raise_on_error=False)
        if before:
            _same(before, after)
        r.append(after)
        s.close()
    _same(r[0], r[2])
    _same(r[1], r[3])
    assert r[0].fmin_lo <= 0.0 <= r[0].fmin_hi   # the minimum of every one of these objectives

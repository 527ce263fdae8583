"""Paper mode (diagonal samples, first-order test on every coordinate) from the
per-parent tables against the interpreter (eval_mode 1): the same run bit for
bit -- sums and products, outer expressions of one and of several variables and
reductions, ragged last blocks, split widths that do not divide a block, both
pools, one and several parents a generation, midpoint and diagonal samples, a
snapshot taken up again, and graph replays."""
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
    if a.n_boxes:
        assert np.array_equal(a.box_lo, b.box_lo) and np.array_equal(a.box_hi, b.box_hi)
        assert np.array_equal(a.box_flo, b.box_flo)
    assert (a.box_evals_fp64, a.mid_evals) == (b.box_evals_fp64, b.mid_evals)


def _solve(p, mode, **opts):
    s = gb.Solver(p, eval_mode=mode, pool_bytes=1 << 30, **opts)
    r = s.solve(raise_on_error=False)
    s.close()
    return r


def _both(p, **opts):
    tab, interp = _solve(p, 0, **opts), _solve(p, 1, **opts)
    _same(tab, interp)
    return tab


FAMS = ["paper_levy", "paper_ackley", "paper_belegundu", "paper_fu", "paper_salomon", "paper_rosenbrock",
        "paper_griewank", "paper_styblinski", "paper_zabinsky", "paper_discontinuous", "paper_rastrigin"]


@pytest.mark.parametrize("fam", FAMS)
@pytest.mark.parametrize("n,B,d", [(7, 5, 5), (11, 5, 3), (4, 4, 2)])
def test_families(fam, n, B, d):
    p = S.make(fam, n=n, block=B)
    _both(p, block=B, split_m=4, split_d=d, max_children=4 ** d, tol_x=1e-2, samples=10, mono_all=1, max_generations=40)


@pytest.mark.parametrize("samples,mono_all", [(1, 1), (0, 1), (3, 0), (64, 1)])
@pytest.mark.parametrize("fam", ["paper_levy", "paper_griewank", "chain", "mixed", "prod_poly"])
def test_options(fam, samples, mono_all):
    n = 13
    p = S.make(fam, n=n, block=4, **({} if fam.startswith("paper") else {"seed": 2}))
    _both(p, block=4, split_m=2, split_d=4, max_children=4 * 16, tol_x=1e-3, samples=samples, mono_all=mono_all,
          max_generations=30)


@pytest.mark.parametrize("fam", ["paper_levy", "paper_ackley", "paper_griewank", "chain"])
@pytest.mark.parametrize("pool_mode", [1, 2])
def test_pools_and_graphs(fam, pool_mode):
    p = S.make(fam, n=20, block=5, **({"seed": 1} if fam == "chain" else {}))
    opts = dict(block=5, split_m=4, split_d=4, max_children=256, tol_x=1e-2, samples=10, mono_all=1, max_generations=50)
    a = _both(p, pool_mode=pool_mode, **opts)
    _same(a, _solve(p, 0, pool_mode=pool_mode, gens_per_sync=4, **opts))


def test_snapshot_taken_up_again():
    p = S.paper_levy(n=10, block=5)
    opts = dict(block=5, split_m=4, split_d=5, max_children=1024, tol_x=1e-4, samples=10, mono_all=1, pool_bytes=1 << 28)
    whole = gb.Solver(p, **opts).solve()
    part = gb.Solver(p, max_generations=4, **opts)
    part.solve(raise_on_error=False)
    rest = gb.Solver(p, **opts).resume(part.snapshot())
    assert rest.generations + 4 == whole.generations
    assert rest.fmin_lo == whole.fmin_lo and rest.fmin_hi == whole.fmin_hi
    assert np.array_equal(rest.box_lo, whole.box_lo) and np.array_equal(rest.box_hi, whole.box_hi)

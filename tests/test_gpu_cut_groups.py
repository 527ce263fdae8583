"""Children cut off in groups of 32 (fan-outs from 2^10 on) against the
interpreter, which evaluates every child at every point: the same run bit for
bit -- fan-outs at and beyond the smallest one that takes groups, ragged last
blocks (fewer children than the fan-out, down to part of one group), several
parents, sums, products, square roots, steps and outer values read from
coordinates; an exponential of a sum takes no groups."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2507_01770_gb300 as gb  # noqa: E402


def _same_run(p, mode, **opts):
    r = []
    for m in (mode, 1):
        s = gb.Solver(p, eval_mode=m, pool_bytes=1 << 30, **opts)
        r.append(s.solve(raise_on_error=False))
        s.close()
    a, b = r
    assert a.status == b.status and a.generations == b.generations
    for k in ("parents", "children", "kept32", "kept", "pool", "gub"):
        assert np.array_equal(a.trace[k], b.trace[k]), k
    assert a.fmin_lo == b.fmin_lo and a.fmin_hi == b.fmin_hi and a.n_boxes == b.n_boxes
    assert np.array_equal(a.box_flo, b.box_flo)
    assert np.array_equal(a.box_lo, b.box_lo) and np.array_equal(a.box_hi, b.box_hi)
    assert (a.box_evals_fp64, a.mid_evals) == (b.box_evals_fp64, b.mid_evals)


# n mod B: 0, 1 (2 or 4 children of a ragged block), 2, B - 1
@pytest.mark.parametrize("n,B,m,d,K", [(20, 10, 2, 10, 1), (25, 12, 2, 11, 3), (11, 5, 4, 5, 2), (17, 5, 4, 5, 1),
                                       (13, 7, 4, 6, 1)])
@pytest.mark.parametrize("fam", ["chain", "sep_cos", "mixed", "paper_fu"])
def test_midpoint_samples(fam, n, B, m, d, K):
    p = S.make(fam, n=n, block=B, **({} if fam.startswith("paper") else {"seed": 3}))
    _same_run(p, 3, block=B, split_m=m, split_d=d, max_children=K * m ** d, max_generations=12, tol_f=1e-6)


@pytest.mark.parametrize("fam", ["paper_levy", "paper_ackley", "paper_salomon", "paper_griewank", "paper_styblinski",
                                 "paper_zabinsky", "paper_discontinuous", "paper_rosenbrock", "prod_poly"])
@pytest.mark.parametrize("n,B,m,d,K", [(11, 5, 4, 5, 1), (12, 10, 2, 10, 2), (8, 6, 4, 6, 1)])
def test_paper_mode(fam, n, B, m, d, K):
    p = S.make(fam, n=n, block=B, **({} if fam.startswith("paper") else {"seed": 2}))
    _same_run(p, 0, block=B, split_m=m, split_d=d, max_children=K * m ** d, tol_x=1e-3, samples=5, mono_all=1,
              max_generations=9)

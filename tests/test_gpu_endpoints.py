"""Children from the endpoint programs (one child per thread, lower and upper
ends only) against the interpreter: the same run bit for bit -- one and several
sums, constants in the outer expression, ragged blocks, split widths that leave
unsplit coordinates in a block, one and several parents a generation, after the
FP32 pass, and both pools.  Objectives the programs do not cover (a nonlinear
outer expression) take the interval walk."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2507_01770_gb300 as gb  # noqa: E402


def _solve(p, mode, **opts):
    s = gb.Solver(p, eval_mode=mode, pool_bytes=1 << 30, **opts)
    r = s.solve(raise_on_error=False)
    s.close()
    return r


@pytest.mark.parametrize("fam", ["chain", "sep_cos", "mixed", "ackley", "paper_rastrigin", "paper_rosenbrock", "paper_fu"])
@pytest.mark.parametrize("n,B,m,d,K", [(33, 10, 2, 7, 1), (21, 10, 4, 4, 5), (40, 20, 2, 6, 3), (130, 10, 4, 5, 1)])
def test_same_run_as_the_interpreter(fam, n, B, m, d, K):
    p = S.make(fam, n=n, block=B, **({} if fam.startswith("paper") else {"seed": 4}))
    for fp32 in (0, 1):
        opts = dict(block=B, split_m=m, split_d=d, max_children=K * m ** d, fp32_prefilter=fp32, max_generations=25,
                    tol_f=1e-6)
        a, b = _solve(p, 3, **opts), _solve(p, 1, **opts)
        assert a.status == b.status and a.generations == b.generations
        for k in ("parents", "children", "kept32", "kept", "pool", "gub"):
            assert np.array_equal(a.trace[k], b.trace[k]), k
        assert a.fmin_lo == b.fmin_lo and a.fmin_hi == b.fmin_hi and a.n_boxes == b.n_boxes
        assert np.array_equal(a.box_flo, b.box_flo)
        assert np.array_equal(a.box_lo, b.box_lo) and np.array_equal(a.box_hi, b.box_hi)
        assert (a.box_evals_fp64, a.mid_evals) == (b.box_evals_fp64, b.mid_evals)

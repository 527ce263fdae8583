"""Children 32 to a block, with the first-order verdicts looked up (objectives
whose sums enter with adjoint [1, 1]) or the outer expression swept per child
(any other, also with coordinates of its own), against the interpreter: the same run bit
for bit -- fan-outs from exactly 32 on, ragged last blocks (fewer valid children
than a block of threads), one and several parents, FP32 first or not, both
pools, launches one by one and replayed, a pool too small for the survivors
(whether they fit is decided after the listing), and more children than the
listing block takes."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2507_01770_gb300 as gb  # noqa: E402


def _same_run(p, **opts):
    r = []
    for mode in (0, 1):
        s = gb.Solver(p, eval_mode=mode, pool_bytes=1 << 28, **opts)
        r.append(s.solve(raise_on_error=False))
        s.close()
    a, b = r
    assert a.status == b.status and a.generations == b.generations
    for k in ("parents", "children", "kept32", "kept", "pool", "gub"):
        assert np.array_equal(a.trace[k], b.trace[k]), k
    assert a.fmin_lo == b.fmin_lo and a.fmin_hi == b.fmin_hi and a.n_boxes == b.n_boxes
    if a.n_boxes:
        assert np.array_equal(a.box_flo, b.box_flo)
        assert np.array_equal(a.box_lo, b.box_lo) and np.array_equal(a.box_hi, b.box_hi)
    assert (a.box_evals_fp32, a.box_evals_fp64, a.mid_evals) == (b.box_evals_fp32, b.box_evals_fp64, b.mid_evals)
    return a


@pytest.mark.parametrize("fam", ["chain", "sep_cos", "mixed", "ackley", "paper_rastrigin", "paper_salomon", "paper_rosenbrock", "paper_levy"])
@pytest.mark.parametrize("fp32", [0, 1])
@pytest.mark.parametrize("n,B,m,d,K", [(23, 10, 2, 5, 16), (21, 10, 2, 10, 1), (19, 9, 2, 6, 3), (13, 6, 4, 3, 4),
                                       (44, 21, 4, 6, 1), (30, 10, 2, 10, 12)])
def test_same_run_as_the_interpreter(fam, fp32, n, B, m, d, K):
    p = S.make(fam, n=n, block=B, **({} if fam.startswith("paper") else {"seed": 7}))
    _same_run(p, block=B, split_m=m, split_d=d, max_children=K * m ** d, fp32_prefilter=fp32, max_generations=40,
              tol_f=1e-6)


@pytest.mark.parametrize("pool_mode", [1, 2])
@pytest.mark.parametrize("sync", [0, 4])
def test_pools_and_replays(pool_mode, sync):
    p = S.mixed(n=150, seed=1, block=15)
    _same_run(p, block=15, split_m=2, split_d=8, max_children=256, fp32_prefilter=1, pool_mode=pool_mode,
              gens_per_sync=sync, max_generations=60, tol_f=1e-6)


@pytest.mark.parametrize("pool_mode", [1, 2])
@pytest.mark.parametrize("K", [1, 3])
def test_survivors_that_do_not_fit(pool_mode, K):
    p = S.chain(n=40, seed=3, block=10)
    a = _same_run(p, block=10, split_m=2, split_d=6, max_children=64 * K, fp32_prefilter=1, pool_mode=pool_mode,
                  max_boxes=48, max_generations=50, tol_f=1e-6)
    assert a.status == gb.GB_E_CAPACITY

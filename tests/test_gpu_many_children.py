"""A generation of more than 2^31 children (parents by the thousand with 2^20
children each), in groups: the same survivors as the walk over every child by
the interpreter."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2507_01770_gb300 as gb  # noqa: E402


def test_more_than_2_31_children():
    K = 3400
    if torch.cuda.mem_get_info()[0] < 160 << 30:
        pytest.skip("needs 160 GB of device memory")
    p = S.chain(n=10, seed=255, block=10)
    r = []
    for mode in (1, 0):
        s = gb.Solver(p, eval_mode=mode, block=10, split_m=4, split_d=10, max_children=K << 20, max_generations=3,
                      pool_bytes=32 << 30, tol_f=56.78)
        r.append(s.solve(device_only=True, raise_on_error=False))
        s.close()
    a, b = r
    for k in ("parents", "children", "kept", "pool", "gub"):
        assert np.array_equal(a.trace[k], b.trace[k]), k
    assert 2048 < a.trace["parents"][-1] < K   # all active regions, in pool order
    assert a.fmin_lo == b.fmin_lo and a.n_boxes == b.n_boxes

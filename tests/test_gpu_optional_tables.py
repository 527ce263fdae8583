"""Tables that only make a solve faster (paper mode's, the child groups'): they
keep to the stated budget, max(64 MiB, pool budget / 8), and a problem that fits
the device without them is created whatever is left for them."""
import ctypes

import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2507_01770_gb300 as gb  # noqa: E402

MIB = 1 << 20
GRAIN = 96 * MIB   # what CUDA's memory pool rounds a problem's memory up by


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _paper(fam, mode, pool, **opts):
    p = S.make(fam, n=30, block=10)
    opts = dict(dict(max_children=1 << 20, max_generations=4), **opts)
    return gb.Solver(p, eval_mode=mode, block=10, split_m=4, split_d=5, samples=10, mono_all=1, tol_x=1e-3,
                     pool_bytes=pool, max_boxes=20000, **opts)


def _held(make):
    f0 = _free()
    s = make()
    held = f0 - _free()
    s.close()
    return held


@pytest.mark.parametrize("fam", ["paper_levy", "paper_griewank", "paper_rastrigin"])
def test_budget_of_the_paper_mode_tables(fam):
    without = _held(lambda: _paper(fam, 1, 1 << 30))
    for pool in (1 << 29, 1 << 30, 2 << 30, 3 << 30, 4 << 30, 5 << 30, 6 << 30, 8 << 30, 12 << 30):
        tables = _held(lambda: _paper(fam, 0, pool)) - without
        assert tables <= max(64 * MIB, pool // 8) + GRAIN, (pool / MIB, tables / MIB)


def _run(s):
    r = s.solve(raise_on_error=False)
    s.close()
    return r


def test_created_without_room_for_the_tables():
    pool = 16 << 30
    gens = dict(max_generations=1 << 20)   # (a million trace rows: 48 MiB beside the tables)
    for _ in range(2):   # (the second time the library's own buffers are in place)
        base = _held(lambda: _paper("paper_levy", 1, pool, **gens))
        full = _held(lambda: _paper("paper_levy", 0, pool, **gens))
    assert full > base + 100 * MIB
    want = _run(_paper("paper_levy", 1, pool, **gens))
    rt = ctypes.CDLL("libcudart.so.13")
    for step in range(25):
        left = base + GRAIN + (full - base) * step // 22
        hog = ctypes.c_void_p()
        assert rt.cudaMalloc(ctypes.byref(hog), ctypes.c_size_t(_free() - left)) == 0
        try:
            r = _run(_paper("paper_levy", 0, pool, **gens))
        finally:
            rt.cudaFree(hog)
        assert r.status == want.status and r.fmin_lo == want.fmin_lo and r.fmin_hi == want.fmin_hi
        assert np.array_equal(r.trace["kept"], want.trace["kept"]) and np.array_equal(r.box_lo, want.box_lo)

"""Creating a problem: the layouts of paper mode's tables take time in
proportion to the objective's length (they are built before a device is looked
for, so this needs none)."""
import time

import pytest

import paper_2507_01770_gb300 as gb
import synthetic as S


def _seconds(p, mode):
    t = time.process_time()
    try:
        gb.Solver(p, eval_mode=mode, block=10, split_m=4, split_d=5, max_children=1 << 10, samples=10, mono_all=1,
                  max_boxes=100).close()
    except gb.GbError as e:
        assert e.status == gb.GB_E_CUDA   # no device here
    return time.process_time() - t


def test_paper_mode_layouts_of_a_long_sum():
    torch = pytest.importorskip("torch")
    if torch.cuda.is_available():
        pytest.skip("times the host part alone")
    p = S.make("paper_levy", n=100_000, block=10)
    runs = [[_seconds(p, m) for m in (0, 1)] for _ in range(3)]   # (processor time: the host may be busy)
    tables, interp = map(min, zip(*runs))
    # the objective itself takes about a second; the layouts must not add half of that
    assert tables < 1.45 * interp, (tables, interp)

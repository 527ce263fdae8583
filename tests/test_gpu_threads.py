"""Host threads with problems of their own, whose kernels need different
amounts of shared memory (all above the 48 KB a launch gets without asking):
no call of one thread may make another's launch fail, and every result is the
one the call gives alone."""
import threading

import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2507_01770_gb300 as gb  # noqa: E402


def _together(jobs, count):
    bar, errs = threading.Barrier(len(jobs)), []

    def run(job):
        try:
            bar.wait()
            for _ in range(count):
                job()
        except Exception as e:   # noqa: BLE001 - reported below
            errs.append(e)

    th = [threading.Thread(target=run, args=(j,)) for j in jobs]
    for t in th:
        t.start()
    for t in th:
        t.join(timeout=300)
    assert not errs, errs


@pytest.mark.parametrize("fp32", [False, True])
def test_box_evaluations(fp32):
    jobs, keep = [], []
    for n in (14000, 24000):   # group sums of 90 and 154 KB
        p = S.chain(n=n, seed=1, block=10)
        s = gb.Solver(p, block=10, pool_bytes=64 << 20)
        lo, hi = S.random_boxes(p, 1, seed=2, around_s=0.5)
        dlo, dhi = torch.from_numpy(lo).cuda(), torch.from_numpy(hi).cuda()
        alone = [t.clone() for t in s.eval_boxes(dlo, dhi, 1, fp32)]
        torch.cuda.synchronize()

        def job(s=s, dlo=dlo, dhi=dhi, alone=alone, out=[t.clone() for t in alone]):
            # (the C call itself: it leaves the interpreter lock, the rest of a pass holds it)
            for _ in range(100):
                rc = gb.load().gb_eval_boxes(s.h.handle, dlo.data_ptr(), dhi.data_ptr(), 1, 1, int(fp32), out[0].data_ptr(),
                                             out[1].data_ptr(), out[2].data_ptr(), out[3].data_ptr(), None)
                assert rc == gb.GB_OK, gb.gb_last_error()
            torch.cuda.synchronize()
            for a, b in zip(alone, out):
                assert torch.equal(a.view(torch.int64) if a.is_floating_point() else a,
                                   b.view(torch.int64) if b.is_floating_point() else b)

        jobs.append(job)
        keep.append(s)
    _together(jobs, 30)
    for s in keep:
        s.close()


@pytest.mark.parametrize("sync", [0, 4])
def test_solves_of_small_fan_out(sync):
    jobs, keep = [], []
    for n in (50, 90):   # blocks of 3, 8 children a parent: several threads per child, 32 children a block
        p = S.chain(n=n, seed=1, block=3)
        s = gb.Solver(p, block=3, split_m=2, split_d=3, max_children=64, max_generations=150, gens_per_sync=sync,
                      pool_bytes=1 << 28)
        alone = s.solve(raise_on_error=False)

        def job(s=s, alone=alone):
            r = s.solve(raise_on_error=False)
            assert r.status == alone.status and r.fmin_lo == alone.fmin_lo and r.fmin_hi == alone.fmin_hi
            for k in ("kept", "pool", "gub"):
                assert np.array_equal(r.trace[k], alone.trace[k])

        jobs.append(job)
        keep.append(s)
    _together(jobs, 40)
    for s in keep:
        s.close()

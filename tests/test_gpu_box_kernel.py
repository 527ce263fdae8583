"""The cooperative box evaluation (several threads per box) at the edges of its
tiles and of the rule that picks the threads per box: sums of 3, 4, 5, 16, 17
and 128 / 129 terms, groups of 128, 129, 512 and 513 terms (the last ones fall
back to one thread per box), blocks of one coordinate, box counts around the
thresholds.  Polynomial objectives: bit for bit the oracle's results."""
import numpy as np
import pytest

import oracle as O
import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2507_01770_gb300 as gb  # noqa: E402


@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("n,B,nbox", [(2, 2, 1), (4, 2, 9), (5, 5, 33), (6, 6, 300), (9, 4, 17), (17, 10, 65), (18, 10, 7),
                                      (33, 32, 2433), (129, 10, 3), (130, 129, 5), (131, 130, 5), (257, 16, 609),
                                      (520, 513, 3), (515, 514, 3), (700, 90, 2)])
def test_box_kernel_bit_exact(n, B, nbox, fp32):
    p = S.chain(n=n, seed=n, block=B)
    s = gb.Solver(p, block=B, pool_bytes=64 << 20)
    orc = O.Oracle(p, block=B)
    lo, hi = S.random_boxes(p, nbox, seed=5, around_s=0.5)
    dlo, dhi = torch.from_numpy(lo).cuda(), torch.from_numpy(hi).cuda()
    nb = (n + B - 1) // B
    pick = sorted(set(np.linspace(0, nbox - 1, min(nbox, 12)).astype(int)))
    for blk in sorted({-1, 0, nb - 1}):
        F, Fm, G, mono = (t.cpu().numpy() for t in s.eval_boxes(dlo, dhi, blk, fp32))
        w = min(B, n - blk * B) if blk >= 0 else 0
        assert np.isnan(G[:, w:]).all()
        for k in pick:
            f, fm, g, m = orc.eval_box(lo[k], hi[k], blk=max(blk, 0), f32=fp32)
            assert np.array_equal(F[k], f) and np.array_equal(Fm[k], fm)
            if blk >= 0:
                assert np.array_equal(G[k, :w], np.asarray(g)[:w]) and mono[k] == m
    s.close()

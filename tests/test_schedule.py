"""The single-frame schedule where whole tiles do not fill the CTAs: whole tiles first, the rest cut in time (CPU)."""
import numpy as np
import pytest


@pytest.mark.parametrize("N,F,T,ctas", [(256, 16, 1024, 152), (250, 61, 4001, 152), (512, 17, 384, 152), (64, 153, 4096, 152),
                                        (64, 151, 4096, 152), (1024, 3, 8000, 152), (300, 7, 16384, 152), (64, 3, 100, 152),
                                        (640, 8, 12800, 10), (128, 1, 128 * 200, 152)])
def test_whole_tiles_then_ranges(N, F, T, ctas):
    import paper_1503_06203_gb300 as xe
    items, grid = xe.plan_schedule(N, F, T, ctas)
    nb, nch = -(-N // 64), -(-T // 128)
    f, bi, bj, c0, c1 = items[:, 0], items[:, 1] & 0xFFFF, items[:, 1] >> 16, items[:, 2], items[:, 3]
    seen = np.zeros((F, nb, nb, nch), dtype=np.int32)
    for k in range(len(items)):
        assert 0 <= c0[k] < c1[k] <= nch
        seen[f[k], bi[k], bj[k], c0[k]:c1[k]] += 1
    iu, ju = np.triu_indices(nb)
    assert (seen[:, iu, ju] == 1).all() and seen.sum() == F * len(iu) * nch
    whole = (c0 == 0) & (c1 == nch)
    n = int(whole.sum())
    assert whole[:n].all() and (n == len(items) or n % ctas == 0)  # whole tiles fill every CTA, then the cut ones
    assert grid == min(ctas, len(items))
    # no CTA has more than the whole-tile schedule would give it
    cost = np.where(bi == bj, 0.7, 1.0) * (c1 - c0) + 0.8
    most = np.bincount(np.arange(len(items)) % grid, weights=cost).max()
    assert most <= -(-F * len(iu) // ctas) * (nch + 0.8) + 1e-9

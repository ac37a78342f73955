"""Schedules where the zeroing of cut tiles' output counts, and the second schedule of frames that are added (CPU, GPU)."""
import numpy as np
import pytest

import oracle
import synth


@pytest.fixture(scope="module")
def xe():
    import paper_1503_06203_gb300 as xe
    xe.build()
    return xe


# a few chunks on an idle GPU: one item a chunk, also where their number is none of the fixed range counts
@pytest.mark.parametrize("N,F,T", [(16, 1, 640), (16, 3, 640), (64, 1, 7 * 128), (64, 2, 11 * 128)])
def test_short_frames_use_a_cta_per_chunk(xe, N, F, T):
    items, grid = xe.plan_schedule(N, F, T, 152)
    assert len(items) == grid == F * (T // 128) and (items[:, 3] - items[:, 2] == 1).all()


# zeroing 71 or 50 MB to spread 32 or 64 tiles takes longer than it gives
@pytest.mark.parametrize("N,F,T", [(1024, 17, 640), (2048, 3, 512)])
def test_large_outputs_are_not_zeroed_for_a_few_tiles(xe, N, F, T):
    items, _ = xe.plan_schedule(N, F, T, 152)
    assert (items[:, 2] == 0).all() and (items[:, 3] == -(-T // 128)).all()


# frames whose first and later frames are scheduled differently, or alike; sums of 8, 16 and 120 bytes modulo 16
@pytest.mark.gpu
@pytest.mark.parametrize("N,F,T", [(1, 1, 700), (5, 1, 5000), (16, 4, 256), (64, 16, 200), (65, 3, 640), (256, 16, 512),
                                   (250, 2, 1000), (512, 1, 8192), (300, 13, 400)])
def test_stored_then_added(xe, N, F, T):
    import torch
    x = synth.uniform(N, F, T, 5 * N + T)
    ref = oracle.visibilities(x)
    xd = torch.from_numpy(x).cuda()
    n = F * xe.baselines(N) * 2
    buf = torch.full((n + 64,), -7, dtype=torch.int32, device="cuda")  # the sums, and what lies behind them
    with xe.Correlator(N, F, T, acc=buf[:n]) as c:
        for _ in range(2):
            for k in (1, 2, 3):
                c.accumulate(xd)
                assert np.array_equal(c.readout().cpu().numpy().astype(np.int64), k * ref), k
            c.reset()
        assert c.status() == 0
    assert (buf[n:] == -7).all()

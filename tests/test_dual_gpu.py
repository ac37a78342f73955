"""The dual-engine correlator kernel (the default share) at the edges of its tiles, chunks and splits, bit-exact.

Whole numbers have one right value, so every comparison is equality (tolerance zero).
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def xe():
    import paper_1503_06203_gb300 as xe
    xe.build()
    return xe


# T around the chunk (128), its k-steps (32) and the dp4a half (64, 96); N around the tile (64), the MMA
# pieces (16, 8) and the dp4a column groups (4); chunk counts past a cycle of the 64/64 and 96/32 splits
@pytest.mark.parametrize("N,F,T", [
    (1, 1, 1), (5, 2, 31), (16, 1, 33), (63, 1, 63), (64, 1, 64), (65, 1, 65), (64, 2, 95), (72, 1, 96),
    (60, 1, 97), (64, 1, 127), (128, 1, 128), (127, 2, 129), (129, 1, 160), (200, 1, 128 * 9 + 70), (64, 1, 128 * 17),
    (192, 300, 40),   # more whole tiles than CTAs, one short chunk each
    (256, 16, 1024),  # whole tiles and time-split ones in one launch
    (20, 1, 128 * 513 + 70), (16, 1, 200000),  # long integrations
])
@pytest.mark.parametrize("extreme", [False, True])
def test_dual_kernel_matches_oracle(xe, N, F, T, extreme):
    import torch
    x = synth.uniform(N, F, T, 7 * N + T)
    if extreme:  # the largest magnitudes: every part -8, or +7 in every other element
        x[:] = 0x00
        x[:, :, 1::2] = 0xFF
        x[T // 2:, :, ::3] = 0x0F
    ref = oracle.visibilities(x)
    xd = torch.from_numpy(x).cuda()
    with xe.Correlator(N, F, T) as c:
        for k in (1, 2):  # stored into a fresh integration, then added onto it
            c.accumulate(xd)
            assert np.array_equal(c.readout().cpu().numpy().astype(np.int64), k * ref), k
        c.reset()
        xe.accumulate_batch([c], [xd])
        assert np.array_equal(c.readout(reset=True).cpu().numpy().astype(np.int64), ref)
        assert c.status() == 0
    if N % 16 == 0:
        out = torch.full((F, xe.baselines(N), 2), -1, dtype=torch.int32, device="cuda")
        xe.correlate_noalloc(xd, out)
        assert np.array_equal(out.cpu().numpy().astype(np.int64), ref)

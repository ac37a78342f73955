"""The lag shift of frames of 16 elements (one quad a row; no repeated ring slot where many CTAs run), bit-exact against the oracle."""
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


# T around a block (128 samples), the ring (8 blocks) and a time segment; lag ranges up to the ring's 512 samples and
# past it; F of a few CTAs, and of more than run at a time (3 on each of 152 SMs)
@pytest.mark.parametrize("F,T", [(1, 1), (2, 63), (3, 128), (1, 1000), (1, 4133), (457, 1), (460, 65), (457, 128), (500, 1025),
                                 (470, 2100)])
@pytest.mark.parametrize("lo,hi", [(0, 0), (-64, 64), (-256, 256), (-257, 256), (300, 300), (-700, 10)])
def test_narrow_frames(xe, F, T, lo, hi):
    import torch
    x = synth.uniform(16, F, T, 3 * T + F)
    lags = np.random.default_rng(T + hi).integers(lo, hi + 1, 16).astype(np.int32)
    lags[3], lags[9] = lo, hi
    y = xe.shift_lags(torch.from_numpy(x).cuda(), torch.from_numpy(lags).cuda())
    assert np.array_equal(y.cpu().numpy(), oracle.shift_lags(x, lags))

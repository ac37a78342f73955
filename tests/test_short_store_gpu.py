"""Frames of one chunk stored by many tiles (the 33 to 128 sample route) and their neighbours, bit-exact against the oracle."""
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


# 303 to 360 tiles (the route starts at two a CTA, 304 on 152), samples around 32 and 128, ragged and unaligned rows
@pytest.mark.parametrize("T", [32, 33, 96, 128, 129])
@pytest.mark.parametrize("N,F", [(64, 303), (64, 304), (130, 60), (256, 31)])
def test_one_chunk_frames(xe, N, F, T):
    import torch
    x = synth.uniform(N, F, T, N + F + T)
    ref = oracle.visibilities(x)
    xd = torch.from_numpy(x).cuda()
    same = lambda v, k: np.array_equal(v.cpu().numpy().astype(np.int64), k * ref)  # noqa: E731
    with xe.Correlator(N, F, T) as a, xe.Correlator(N, F, T) as b:
        for k in (1, 2):  # stored, then added onto
            a.accumulate(xd)
            assert same(a.readout(), k)
        xe.accumulate_batch([a, b], [xd, xd])  # one added onto, one stored
        assert same(a.readout(reset=True), 3) and same(b.readout(reset=True), 1)
        xe.accumulate_batch([a, b], [xd, xd])  # both stored
        assert same(a.readout(), 1) and same(b.readout(), 1)
        assert a.status() == 0 and b.status() == 0
    if N % 16 == 0:
        out = torch.full((F, xe.baselines(N), 2), -1, dtype=torch.int32, device="cuda")
        xe.correlate_noalloc(xd, out)
        assert same(out, 1)

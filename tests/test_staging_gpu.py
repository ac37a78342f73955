"""Frames whose rows are not 16-byte aligned (copied into a staging buffer first), bit-exact against the oracle."""
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


@pytest.mark.parametrize("N,F,T", [(1, 1, 1), (1, 3, 5), (3, 2, 130), (15, 1, 64), (17, 5, 77), (31, 1, 300), (66, 3, 129),
                                   (250, 2, 200), (1000, 1, 33)])
@pytest.mark.parametrize("shift", [0, 1, 6, 15])
def test_unaligned_rows(xe, N, F, T, shift):
    import torch
    x = synth.uniform(N, F, T, 100 + N + shift)
    flat = torch.zeros(shift + x.size, dtype=torch.uint8, device="cuda")
    flat[shift:] = torch.from_numpy(x.reshape(-1)).cuda()
    xd = flat[shift:].view(T, F, N)  # contiguous, its first byte `shift` past an aligned one
    with xe.Correlator(N, F, T) as c:
        c.accumulate(xd)
        assert np.array_equal(c.readout().cpu().numpy().astype(np.int64), oracle.visibilities(x))
    if F > 1:  # a band range of it
        with xe.Correlator(N, F, T, bands=(1, F)) as c:
            c.accumulate(xd)
            assert np.array_equal(c.readout().cpu().numpy().astype(np.int64), oracle.visibilities(np.ascontiguousarray(x[:, 1:])))


def test_aligned_rows_at_an_unaligned_address(xe):
    import torch
    N, F, T = 64, 3, 200
    x = synth.uniform(N, F, T, 5)
    flat = torch.zeros(5 + x.size, dtype=torch.uint8, device="cuda")
    flat[5:] = torch.from_numpy(x.reshape(-1)).cuda()
    with xe.Correlator(N, F, T) as c:
        c.accumulate(flat[5:].view(T, F, N))
        assert np.array_equal(c.readout().cpu().numpy().astype(np.int64), oracle.visibilities(x))

"""Gated correlation whose runs of samples start anywhere: run lengths around the chunk, cut first and last runs,
gates without positions or samples, bit-exact against the oracle (whole numbers: tolerance zero)."""
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


@pytest.mark.parametrize("N,F,T,G,period,phase", [
    (64, 1, 1000, 1, 130, 7),      # one gate: every sample, whatever the period
    (80, 2, 1500, 2, 254, 13),     # runs of 127
    (64, 1, 1500, 2, 256, 255),    # runs of 128, the first one sample long
    (64, 1, 1500, 2, 258, 1),      # runs of 129
    (65, 1, 1111, 3, 700, 699),    # runs of several chunks and a rest
    (64, 2, 900, 8, 128, 5),       # runs of 16
    (48, 1, 400, 130, 129, 60),    # more gates than positions
    (64, 1, 129, 4, 512, 511),     # gates without samples
    (130, 3, 2048, 8, 1024, 100),
])
def test_gate_runs(xe, N, F, T, G, period, phase):
    import torch
    x = synth.uniform(N, F, T, 11 * G + period)
    gates = [xe.Correlator(N, F, T) for _ in range(G)]
    ref = oracle.gated(x, G, period, phase)
    xd = torch.from_numpy(x).cuda()
    for k in (1, 2):
        xe.accumulate_gated(gates, xd, period, phase)
        for g, c in enumerate(gates):
            assert np.array_equal(c.readout().cpu().numpy().astype(np.int64), k * ref[g]), (k, g)
    assert gates[0].status() == 0

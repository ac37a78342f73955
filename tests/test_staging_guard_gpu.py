"""What lies around an unaligned frame never shows in its result: guard bytes of several values on both sides."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,F,T", [(1, 1, 1), (2, 1, 3), (17, 1, 1), (33, 2, 5), (250, 3, 129)])
def test_guard_bytes(N, F, T):
    import torch
    import paper_1503_06203_gb300 as xe
    xe.build()
    x = synth.uniform(N, F, T, 9 * N + T)
    ref = oracle.visibilities(x)
    with xe.Correlator(N, F, T) as c:
        for guard in (0x00, 0x88, 0xFF):
            for shift in (1, 2, 3, 4):
                flat = torch.full((shift + x.size + 4,), guard, dtype=torch.uint8, device="cuda")
                flat[shift:shift + x.size] = torch.from_numpy(x.reshape(-1)).cuda()
                c.accumulate(flat[shift:shift + x.size].view(T, F, N))
                assert np.array_equal(c.readout(reset=True).cpu().numpy().astype(np.int64), ref), (guard, shift)

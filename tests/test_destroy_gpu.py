"""Destroying a handle whose last call was captured leaves no error for the next handle's launches."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def test_destroy_after_capture():
    import torch
    import paper_1503_06203_gb300 as xe
    xe.build()
    shapes = [(256, 4, 1024), (64, 4, 2048), (50, 3, 500), (64, 4, 2048)]
    st = torch.cuda.Stream()
    for N, F, T in shapes:
        x = synth.uniform(N, F, T, N + T)
        xd = torch.from_numpy(x).cuda()
        out = torch.zeros(F, xe.baselines(N), 2, dtype=torch.int32, device="cuda")
        with xe.Correlator(N, F, T) as c:
            with torch.cuda.stream(st):
                st.wait_stream(torch.cuda.default_stream())
                c.accumulate(xd)
                st.synchronize()
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=st):
                    c.accumulate(xd)
                    c.readout(out)
                g.replay()
                st.synchronize()
            assert np.array_equal(out.cpu().numpy().astype(np.int64), 2 * oracle.visibilities(x))
            del g

"""Captured calls of the cycle-popping sampler: sized by a call of any graph of
the device, as the walker kernels' shared buffer is."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

fc = pytest.importorskip("paper_2101_06192_gb300.fc")


def test_capture_after_a_call_of_another_graph():
    """Tree state beyond shared memory: an uncaptured call of any live graph of
    the device is enough, as for the walker kernels' shared buffer."""
    g = synth.barabasi_albert(40001, 4, 2)
    tau = 8
    with fc.Graph.from_csr(g, [1.0]) as A, fc.Graph.from_csr(g, [1.0]) as B:
        ref = A.sample(3, tau, with_C=False)["R"]
        assert A.last_kernel() == 5
        R = torch.zeros(g.n, dtype=torch.int32, device="cuda")
        s = torch.cuda.Stream()
        cg = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            with torch.cuda.graph(cg, stream=s):
                R.zero_()
                B.sample_async(3, tau, R, stream=s)
        for _ in range(2):
            cg.replay()
            torch.cuda.synchronize()
            B.check()
            assert torch.equal(R, ref)

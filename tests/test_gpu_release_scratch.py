"""fc_release_scratch gives back what the cycle-popping sampler took."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

fc = pytest.importorskip("paper_2101_06192_gb300.fc")

MB = 1 << 20


def test_release_gives_the_pool_back():
    """2^18 vertices x 64 trees: 268 MB of scratch, held by the pool after the
    call until it is released."""
    g = synth.torus(512, 512)
    with fc.Graph.from_csr(g, [1.0]) as G:
        R = torch.zeros(g.n, dtype=torch.int32, device="cuda")
        assert fc.lib().fc_release_scratch() == 0
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        G.sample(3, 64, R=R, with_C=False)
        assert G.last_kernel() == 5
        torch.cuda.synchronize()
        assert before - torch.cuda.mem_get_info()[0] > 200 * MB
        assert fc.lib().fc_release_scratch() == 0
        assert before - torch.cuda.mem_get_info()[0] < 64 * MB
        again = G.sample(3, 64, with_C=False)["R"]
    assert torch.equal(again, R)

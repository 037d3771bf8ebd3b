"""Parents alone take the automatic sampler at every size (cycle popping), and
equal the edge-record kernel's."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

fc = pytest.importorskip("paper_2101_06192_gb300.fc")


@pytest.mark.parametrize("n", [(1 << 15) + 1, 50_000, 1 << 16])
def test_parents_come_from_the_automatic_sampler(n):
    g = synth.barabasi_albert(n, 4, 2)
    with fc.Graph.from_csr(g, [1.0]) as G:
        outs = []
        for k in (0, 2):
            G.set_kernel(k)
            outs.append(G.sample(3, 6, want_parents=True))
            assert (G.last_kernel() == 5) == (k == 0)
        for key in ("parents", "R", "C"):
            assert torch.equal(outs[0][key], outs[1][key]), key

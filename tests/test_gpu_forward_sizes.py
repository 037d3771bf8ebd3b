"""The network's forward pass at the sizes where its vertices per thread change
(1, 2, 4 and 8 from 77,824, 155,648 and 311,296 vertices on), against the oracle."""
import numpy as np
import pytest
import torch

import synth
from oracle import cv as ocv

pytestmark = pytest.mark.gpu

fc = pytest.importorskip("paper_2101_06192_gb300.fc")


@pytest.mark.parametrize("n", [1, 77823, 77824, 155647, 155649, 311295, 311296, 312321])
def test_forward_at_tile_edges(n):
    g = synth.path(n)
    rng = np.random.default_rng(n)
    X = rng.normal(size=(n, 4)).astype(np.float32)
    p32 = rng.normal(scale=0.5, size=769).astype(np.float32)
    params = torch.from_numpy(p32).cuda()
    with fc.Graph.from_csr(g, [1.0]) as G:
        out = G.mlp_forward(torch.from_numpy(X).cuda(), params).cpu().numpy()
    pb = params.to(torch.bfloat16).to(torch.float64).cpu().numpy()
    po = {"W1": pb[:512].reshape(128, 4), "b1": pb[512:640], "w2": pb[640:768], "b2": pb[768]}
    pre = X.astype(np.float64) @ po["W1"].T + po["b1"]
    z = np.maximum(pre, 0.0) @ po["w2"] + po["b2"]
    p = ocv.p_root(g, 1.0)
    ref = p + (1.0 - p) / (1.0 + np.exp(-z))
    # 640 FP32 roundings of partial sums of size up to |z| terms: 1e-4 of z at most, through a slope of 1/4
    np.testing.assert_allclose(out, ref, rtol=0, atol=2e-5 * (1.0 + np.abs(pre).max()))

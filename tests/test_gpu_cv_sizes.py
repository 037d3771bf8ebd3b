"""Neighbour-degree sums at the edges of a tile of CSR entries, and the
network passes at odd numbers of vertices and with features that are not finite,
against the FP64 oracle (tolerances of tests/test_gpu_cv.py)."""
import numpy as np
import pytest
import torch

import synth
from oracle import cv as ocv
from oracle import mlp
from test_gpu_cv import _from_oracle, _to_oracle

pytestmark = pytest.mark.gpu

fc = pytest.importorskip("paper_2101_06192_gb300.fc")
cvnet = pytest.importorskip("paper_2101_06192_gb300.cvnet")


@pytest.mark.parametrize("kind", ["one", "edge", "star1025", "star1026", "star9000", "path1025", "isolated", "hubs"])
def test_neighbour_degree_sums(kind):
    """2048 and 2050 entries, a row over five tiles, long runs of empty rows."""
    g = {"one": lambda: synth.empty(3), "edge": lambda: synth.path(2), "star1025": lambda: synth.star(1025),
         "star1026": lambda: synth.star(1026), "star9000": lambda: synth.star(9000), "path1025": lambda: synth.path(1025),
         "isolated": lambda: synth.from_edges(50000, *synth.barabasi_albert(400, 2, 9).edges()[:2]),
         "hubs": lambda: synth.barabasi_albert(20000, 7, 3)}[kind]()
    with fc.Graph.from_csr(g, [0.7]) as G:
        np.testing.assert_allclose(G.features().cpu().numpy(), mlp.features(g, 0.7), rtol=2e-6, atol=2e-6)


def _case(n, seed):
    g = synth.path(n) if n < 8 else synth.barabasi_albert(n, 3, seed)
    Xo = mlp.features(g, 1.0)
    rng = np.random.default_rng(seed)
    p = ocv.p_root(g, 1.0)
    y = np.clip(p + 0.3 * rng.random(g.n), 0, 1).astype(np.float32)
    params = cvnet.init_params(11)
    torch.manual_seed(seed)
    params += 0.05 * torch.randn_like(params)
    return g, Xo.astype(np.float32), p, y, params


@pytest.mark.parametrize("n", [1, 2, 127, 128, 129, 255, 256, 257, 1023, 1025, 80001, 160001])
def test_network_at_odd_sizes(n):
    """One, two (80001) and four (160001) vertices per thread of the gradient pass."""
    g, X, p, y, params = _case(n, n)
    po = _to_oracle(params.cpu().numpy())
    with fc.Graph.from_csr(g, [1.0]) as G:
        loss, grad = G.mlp_loss_grad(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), params)
        out = G.mlp_forward(torch.from_numpy(X).cuda(), params).cpu().numpy()
    l_ref, g_ref = mlp.loss_and_grads(po, X.astype(np.float64), p, y.astype(np.float64))
    gr = _from_oracle(g_ref)
    assert abs(float(loss.item()) - l_ref) <= 1e-4 * abs(l_ref)
    np.testing.assert_allclose(grad.cpu().numpy().astype(np.float64), gr, rtol=2e-3, atol=2e-4 * np.abs(gr).max())
    ref, _ = mlp.forward(po, X.astype(np.float64), p)
    np.testing.assert_allclose(out, ref, rtol=1e-5, atol=1e-6)


@pytest.mark.parametrize("v", [0, 130, 255])
def test_features_that_are_not_finite(v):
    """No unit is active for a vertex whose features are NaN: it adds nothing
    to the hidden layer's gradient."""
    g, X, p, y, params = _case(256, 5)
    X[v] = np.nan
    keep = np.arange(256) != v
    po = _to_oracle(params.cpu().numpy())
    with fc.Graph.from_csr(g, [1.0]) as G:
        _, grad = G.mlp_loss_grad(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), params)
    _, g_ref = mlp.loss_and_grads(po, X[keep].astype(np.float64), p[keep], y[keep].astype(np.float64))
    gr = _from_oracle(g_ref)[:768] * (255 / 256)
    np.testing.assert_allclose(grad.cpu().numpy().astype(np.float64)[:768], gr, rtol=2e-3, atol=2e-4 * np.abs(gr).max())

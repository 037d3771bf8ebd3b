"""The CG from a start of zeros (its first residual is b) and from others, and
group closeness over two batches of columns."""
import numpy as np
import pytest
import torch

import synth
from oracle import dense

pytestmark = pytest.mark.gpu

fc = pytest.importorskip("paper_2101_06192_gb300.fc")


@pytest.mark.parametrize("m", [1, 3, 65, 129, 131])
@pytest.mark.parametrize("start", ["zero", "minus_zero", "last_entry", "solution", "random"])
def test_start(m, start):
    """Error at most 1e-12 |b| per column, as from any start."""
    g = synth.barabasi_albert(301, 3, 9, weighted=True)
    om = dense.forest_matrix(g, 0.7)
    rng = np.random.default_rng(m)
    b = rng.standard_normal((m, g.n))
    x = torch.zeros(m, g.n, dtype=torch.float64, device="cuda")
    if start == "minus_zero":
        x.neg_()
    elif start == "last_entry":
        x[-1, -1] = 1e3
    elif start == "solution":
        x.copy_(torch.from_numpy(b @ om))
    elif start == "random":
        x.copy_(torch.from_numpy(rng.standard_normal((m, g.n))))
    with fc.Graph.from_csr(g, [0.7]) as G:
        x, it = G.solve(torch.from_numpy(b).cuda(), x=x, rel_tol=1e-12)
    if start == "solution":
        assert it == 0
    err = np.linalg.norm(x.cpu().numpy() - b @ om, axis=1)
    assert np.all(err <= 2e-12 * np.linalg.norm(b, axis=1) + 1e-15), err.max()


def test_group_over_two_batches():
    """n = 4101: batches of 2176 and 1925 columns (the last filled up)."""
    g = synth.barabasi_albert(4101, 3, 2)
    om = dense.forest_matrix(g, 1.0)
    k = 4
    with fc.Graph.from_csr(g, [1.0]) as G:
        S, far = G.group_closeness(k, rel_tol=1e-12)
    S = [int(v) for v in S]
    n = g.n
    full = np.zeros((n + 1, n + 1))
    full[:n, :n] = om
    v0 = int(np.argmin(np.diag(om)))
    M = full - full[:, [v0]] - full[[v0], :] + full[v0, v0]
    M[v0, :] = M[:, v0] = 0.0
    assert S[0] == v0
    for i in range(1, k):
        np.testing.assert_allclose(float(far[i - 1]), np.trace(M), rtol=1e-9)
        gain = np.where(np.diag(M)[:n] > 0, (M[:, :n] ** 2).sum(axis=0) / np.maximum(np.diag(M)[:n], 1e-300), -1.0)
        gain[S[:i]] = -1.0
        assert gain[S[i]] >= gain.max() * (1 - 1e-9)
        m = M[S[i]].copy()
        M -= np.outer(m, m) / m[S[i]]
        M[S[i], :] = M[:, S[i]] = 0.0
    np.testing.assert_allclose(float(far[k - 1]), np.trace(M), rtol=1e-9)

"""Laplacian solves around the length up to which columns are centred in one
launch (8192 entries), one and several columns, against the definition of L^+ b."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

fc = pytest.importorskip("paper_2101_06192_gb300.fc")


def _graph(n):
    return {2: lambda: synth.path(2), 257: lambda: synth.complete(257), 8192: lambda: synth.torus(64, 128),
            8193: lambda: synth.barabasi_albert(8193, 3, 1)}[n]()


@pytest.mark.parametrize("n", [2, 257, 8192, 8193])
@pytest.mark.parametrize("m", [1, 3, 40])
def test_mean_zero_solution(n, m):
    g = _graph(n)
    rng = np.random.default_rng(n + m)
    b = rng.normal(size=(m, n))
    with fc.Graph.rooted(g, 0) as G:
        x, _ = G.laplacian_solve(torch.from_numpy(b).cuda(), rel_tol=1e-11)
    x = x.cpu().numpy()
    row = np.repeat(np.arange(n), np.diff(g.rowptr))
    w = np.ones(g.nnz) if g.w is None else g.w.astype(np.float64)
    d = np.bincount(row, w, minlength=n)
    for j in range(m):
        r = b[j] - b[j].mean() - (d * x[j] - np.bincount(row, w * x[j][g.colidx], minlength=n))
        # the solver's own tolerance and the rounding of this residual
        assert np.linalg.norm(r) <= 1e-10 * np.linalg.norm(b[j])
        assert abs(x[j].mean()) <= 1e-12 * (1.0 + np.abs(x[j]).max())


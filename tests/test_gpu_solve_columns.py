"""Several right-hand sides of the CG at the widths and row lengths where the
interleaved kernels change form: lanes per row (2..32), values per lane (1, 2,
4), rows around a segment's length, empty rows; against the oracle's CG.  The
refinement stops at a relative FP64 residual of 1e-12 and every eigenvalue of
I + alpha L is at least 1, so the error is at most 1e-12 |b| per column."""
import numpy as np
import pytest
import torch

import synth
from oracle import dense

pytestmark = pytest.mark.gpu

fc = pytest.importorskip("paper_2101_06192_gb300.fc")


def _hubs(weighted):
    """Hub rows of 63..65, 127..129, 256 and 300 entries, vertices without edges."""
    u, v = [], []
    for i, d in enumerate((63, 64, 65, 127, 128, 129, 256, 300)):
        u += [i] * d
        v += list(range(8, 8 + d))
    w = None if not weighted else np.random.default_rng(3).uniform(1, 10, len(u)).astype(np.float32)
    return synth.from_edges(340, np.array(u), np.array(v), w)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("m", [2, 3, 4, 5, 8, 9, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 130, 132])
def test_columns_against_dense_inverse(m, weighted):
    g = _hubs(weighted)
    om = dense.forest_matrix(g, 0.7)
    rng = np.random.default_rng(m)
    b = rng.standard_normal((m, g.n))
    b[0] = 0.0  # a column that is solved from the start
    with fc.Graph.from_csr(g, [0.7]) as G:
        x, _ = G.solve(torch.from_numpy(b).cuda(), rel_tol=1e-12)
        again, _ = G.solve(torch.from_numpy(b).cuda(), rel_tol=1e-12)
    assert torch.equal(x, again)
    ref = b @ om
    err = np.linalg.norm(x.cpu().numpy() - ref, axis=1)
    assert np.all(err <= 2e-12 * np.linalg.norm(b, axis=1) + 1e-15), err.max()


@pytest.mark.parametrize("m", [1, 2, 7, 40])
def test_laplacian_columns(m):
    """Mean-projected columns of L^+ (column-major and interleaved)."""
    from oracle import electrical as el
    g = synth.barabasi_albert(777, 3, 9, weighted=True)
    root = int(np.argmax(g.degrees()))
    lp = el.laplacian_pinv(g)
    b = np.random.default_rng(m).standard_normal((m, g.n))
    with fc.Graph.rooted(g, root) as G:
        x, _ = G.laplacian_solve(torch.from_numpy(b).cuda(), rel_tol=1e-12)
    ref = (b - b.mean(axis=1, keepdims=True)) @ lp
    lam = np.linalg.norm(lp, 2)  # 1 / the smallest non-zero eigenvalue
    err = np.linalg.norm(x.cpu().numpy() - ref, axis=1)
    assert np.all(err <= 2e-12 * lam * np.linalg.norm(b, axis=1) + 1e-13 * np.linalg.norm(ref, axis=1)), err.max()

"""Rao-Blackwellised sums at the edges of the kernel's chunks:
1 to 33 trees, n around a chunk of 1024 vertices, rows of one segment and one
entry more, deep trees; bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import synth
from oracle import rb

pytestmark = pytest.mark.gpu

fc = pytest.importorskip("paper_2101_06192_gb300.fc")


def _check(g, alpha, tau, seed=5):
    with fc.Graph.from_csr(g, [alpha]) as G:
        par = G.sample(seed, tau, want_parents=True)["parents"][0]
        acc = G.rb_accumulate(par)
    np.testing.assert_array_equal(acc.cpu().numpy().view(np.uint64), rb.accumulate(g, alpha, par.cpu().numpy()))


@pytest.mark.parametrize("n", [1, 2, 33, 1023, 1024, 1025, 2049])
@pytest.mark.parametrize("tau", [1, 5, 31, 32, 33])
def test_sizes(n, tau):
    _check(synth.path(n) if n < 40 else synth.barabasi_albert(n, 3, n), 1.5, tau)


@pytest.mark.parametrize("d", [255, 256, 257, 512, 513])
@pytest.mark.parametrize("weighted", [False, True])
def test_rows_around_a_segment(d, weighted):
    u, v = np.zeros(d, np.int64), np.arange(1, d + 1)
    w = np.random.default_rng(d).uniform(0.5, 2.0, d).astype(np.float32) if weighted else None
    _check(synth.from_edges(d + 3, u, v, w), 0.8, 9)


@pytest.mark.parametrize("name", ["path", "grid"])
def test_deep_trees(name):
    """Paths of thousands of vertices to u* (a large alpha)."""
    _check(synth.path(5000) if name == "path" else synth.perturbed_grid(60, 51, 3), 1e4, 7)

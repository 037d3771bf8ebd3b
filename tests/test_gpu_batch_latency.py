"""Per-graph completion times of a batch (fc_batch_latency) under the
cycle-popping sampler: a graph is complete when the last cycle of its last
tree is found, not when the launch ends."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

fc = pytest.importorskip("paper_2101_06192_gb300.fc")

POP = 5


def _batch():
    """Graphs of a few vertices around one whose cycles take many rounds."""
    graphs = [synth.path(5), synth.empty(3), synth.torus(120, 121), synth.complete(6)]
    u, offs = synth.union(graphs)
    return u, offs, np.array([0.5, 1.0, 60.0, 0.1])


def test_small_graphs_complete_before_a_large_one():
    """16 trees (one CTA each): the small graphs' stamps come after the drawing
    or an early round, the large one's after its last round."""
    u, offs, alphas = _batch()
    with fc.Graph.batch(u, offs, alphas) as G:
        for _ in range(2):
            G.sample(7, 16, want_visits=True)
            assert G.last_kernel() == POP
            lat = G.batch_latency_ms()
            assert np.all(lat > 0)
            for small in (0, 1, 3):
                assert lat[small] < 0.5 * lat[2], lat


def test_parents_are_part_of_the_trees():
    """With parents a tree is complete when its row of them is written."""
    u, offs, alphas = _batch()
    with fc.Graph.batch(u, offs, alphas) as G:
        G.sample(7, 16, want_parents=True)
        assert G.last_kernel() == POP
        lat = G.batch_latency_ms()
        assert np.all(lat > 0.5 * lat[2]), lat

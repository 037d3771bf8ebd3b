"""The cycle-popping sampler (the automatic choice) against the oracle and the
walker kernels: trees, counts, departures and step counts bit-exact, at the
edges of its chunks, rows, windows and teams."""
import numpy as np
import pytest
import torch

import synth
from oracle import native

pytestmark = pytest.mark.gpu

fc = pytest.importorskip("paper_2101_06192_gb300.fc")

POP = 5


def _u32(t):
    return t.cpu().numpy().view(np.uint32)


def _check(G, g, alphas, seed, tau, tree_offset=0):
    out = G.sample(seed, tau, tree_offset=tree_offset, want_parents=True, want_steps=True, want_visits=True)
    assert G.last_kernel() == POP
    n = g.n
    for a, al in enumerate(alphas):
        ref = native.wilson(g, al, seed=seed, tau=tau, tree_offset=tree_offset, alpha_idx=a, want_parents=True,
                            want_visits=True)
        np.testing.assert_array_equal(out["parents"][a].cpu().numpy(), ref["parents"])
        np.testing.assert_array_equal(_u32(out["R"]).reshape(-1, n)[a], ref["R"])
        np.testing.assert_array_equal(_u32(out["C"]).reshape(-1, n)[a], ref["C"])
        np.testing.assert_array_equal(out["steps"][a].cpu().numpy().astype(np.uint64), ref["steps"])
        np.testing.assert_array_equal(out["visits"].view(-1, n)[a].cpu().numpy().astype(np.uint64), ref["visits"])
    return out


@pytest.mark.parametrize("n", [1, 2, 31, 255, 256, 257, 1000, 4099])
@pytest.mark.parametrize("weighted", [False, True])
def test_sizes_bit_exact(n, weighted):
    """Below, at and above a warp's chunk of 256 vertices and rows that are not
    a multiple of four words; 1, 5 and 33 trees (fewer trees than teams, rows
    that do not divide evenly)."""
    g = synth.random_small(n, 0.5, 3, weighted) if n < 32 else synth.erdos_renyi(n, 6, 3, weighted=weighted)
    with fc.Graph.from_csr(g, [0.3, 5.0]) as G:
        for tau in (1, 5, 33):
            _check(G, g, [0.3, 5.0], 11, tau, tree_offset=tau)


@pytest.mark.parametrize("name", ["empty", "star", "path", "K8", "isolated", "torus", "grid", "ba_hubs", "ba_weighted",
                                  "rmat"])
def test_shapes_bit_exact(name):
    """Long cycles (path, torus at a large alpha), hubs whose rows exceed the
    eight thresholds kept in registers, vertices without edges."""
    alphas = [0.5, 40.0]
    g = {"empty": lambda: synth.empty(37), "star": lambda: synth.star(300), "path": lambda: synth.path(500),
         "K8": lambda: synth.complete(8), "torus": lambda: synth.torus(64, 65),
         "isolated": lambda: synth.from_edges(1000, *synth.barabasi_albert(400, 2, 9).edges()[:2]),
         "grid": lambda: synth.perturbed_grid(60, 51, 3), "ba_hubs": lambda: synth.barabasi_albert(20000, 7, 3),
         "ba_weighted": lambda: synth.barabasi_albert(3000, 5, 3, weighted=True),
         "rmat": lambda: synth.rmat(11, 16, 4)}[name]()
    with fc.Graph.from_csr(g, alphas) as G:
        _check(G, g, alphas, 5, 21)


@pytest.mark.parametrize("name", ["path", "ba", "ba_weighted", "torus"])
def test_rooted_bit_exact(name):
    g = {"path": lambda: synth.path(200), "ba": lambda: synth.barabasi_albert(4001, 3, 5),
         "ba_weighted": lambda: synth.barabasi_albert(900, 4, 5, weighted=True),
         "torus": lambda: synth.torus(20, 21)}[name]()
    root = int(np.argmax(g.degrees()))
    tau = 19
    with fc.Graph.rooted(g, root) as G:
        out = G.sample(8, tau, want_parents=True, want_steps=True, want_visits=True, with_C=False)
        assert G.last_kernel() == POP
    ref = native.wilson_rooted(g, root, seed=8, tau=tau, want_visits=True)
    np.testing.assert_array_equal(out["parents"][0].cpu().numpy(), ref["parents"])
    np.testing.assert_array_equal(out["steps"][0].cpu().numpy().astype(np.uint64), ref["steps"] + 1)
    vis = ref["visits"].copy()
    vis[root] = tau
    np.testing.assert_array_equal(out["visits"].cpu().numpy().astype(np.uint64), vis)


def test_batch_bit_exact():
    graphs, alphas = synth.uneven_batch(23, 5, n_min=1, n_max=700)
    u, offs = synth.union(graphs)
    with fc.Graph.batch(u, offs, alphas) as G:
        out = G.sample(9, 13, want_parents=True, want_steps=True, want_visits=True)
        assert G.last_kernel() == POP
        lat = G.batch_latency_ms()
    ref = native.wilson(u, np.repeat(alphas, np.diff(offs)), seed=9, tau=13, want_parents=True, want_visits=True)
    np.testing.assert_array_equal(out["parents"][0].cpu().numpy(), ref["parents"])
    np.testing.assert_array_equal(_u32(out["R"]), ref["R"])
    np.testing.assert_array_equal(_u32(out["C"]), ref["C"])
    np.testing.assert_array_equal(out["visits"].cpu().numpy().astype(np.uint64), ref["visits"])
    steps = out["steps"].cpu().numpy()  # [graph][tree]
    np.testing.assert_array_equal(steps.sum(axis=0).astype(np.uint64), ref["steps"])
    assert np.all(steps >= np.diff(offs)[:, None]) and np.all(lat > 0)


def test_several_windows_equal_walker_kernel():
    """Two windows per team and rows of two alphas in one window: counts,
    departures and steps equal the edge-record kernel's."""
    g = synth.barabasi_albert((1 << 20) - 3, 4, 2)
    with fc.Graph.from_csr(g, [1.0, 0.2]) as G:
        outs = []
        for k in (0, 2):
            G.set_kernel(k)
            outs.append(G.sample(6, 170, want_steps=True, want_visits=True))
            assert (G.last_kernel() == POP) == (k == 0)
        for key in ("R", "C", "visits", "steps"):
            assert torch.equal(outs[0][key], outs[1][key]), key
        G.set_kernel(0)
        again = G.sample(6, 170, want_steps=True, want_visits=True)
        for key in ("R", "C", "visits", "steps"):
            assert torch.equal(outs[0][key], again[key]), key


def test_watchdog_and_context():
    """A budget of a few steps ends the call with FC_ETIMEOUT; the next call is
    whole again."""
    g = synth.torus(40, 41)
    with fc.Graph.from_csr(g, [30.0]) as G:
        with pytest.raises(fc.FcError) as e:
            G.sample(3, 8, max_steps_per_tree=5)
        assert e.value.status == fc.FC_ETIMEOUT
        _check(G, g, [30.0], 3, 8)


def test_capture_needs_a_sized_call():
    """As for the walker kernels, a graph whose tree state exceeds shared memory
    is captured only after an uncaptured call; the replay equals it."""
    g = synth.barabasi_albert(40001, 4, 2)
    tau = 8
    with fc.Graph.from_csr(g, [1.0]) as G:
        R = torch.zeros(g.n, dtype=torch.int32, device="cuda")
        s = torch.cuda.Stream()
        cg = torch.cuda.CUDAGraph()
        with torch.cuda.stream(s):
            with pytest.raises(fc.FcError):
                with torch.cuda.graph(cg, stream=s):
                    G.sample_async(3, tau, R, stream=s)
        torch.cuda.synchronize()
        ref = G.sample(3, tau, with_C=False)["R"]
        cg = torch.cuda.CUDAGraph()
        with torch.cuda.stream(s):
            with torch.cuda.graph(cg, stream=s):
                R.zero_()
                G.sample_async(3, tau, R, stream=s)
        for _ in range(2):
            cg.replay()
            torch.cuda.synchronize()
            G.check()
            assert torch.equal(R, ref)

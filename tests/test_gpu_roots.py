"""Forest roots and depths: pointer jumping (chunk edges, several windows, deep
trees) against plain doubling on the CPU, and the sampler's automatic forest
outputs against the edge-record kernel's, which records them as vertices join."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

fc = pytest.importorskip("paper_2101_06192_gb300.fc")


def _ref(par):
    T, n = par.shape
    own = np.arange(n)[None, :]
    anc = np.where(par == n, own, par)
    dep = (par != n).astype(np.int64)
    for _ in range(32):
        dep = dep + np.take_along_axis(dep, anc, 1)
        anc = np.take_along_axis(anc, anc, 1)
    return anc, dep


@pytest.mark.parametrize("n,T", [(1, 1), (1, 300), (255, 2), (1023, 3), (1024, 1), (1025, 5), (4096, 2), (70001, 3),
                                 (5000, 3500), (9000001, 2)])
def test_pointer_jumping(n, T):
    """3500 trees of 5000 vertices and 2 of 9000001 are several windows each."""
    rng = np.random.default_rng(n)
    par = np.minimum((rng.random((T, n)) * np.arange(n)[None, :]).astype(np.int64), np.arange(n) - 1)
    par[rng.random((T, n)) < 0.01] = n
    par[:, 0] = n
    par[0, 1:] = np.arange(n - 1)  # a path
    perm = rng.permutation(n)
    inv = np.append(perm, n)  # vertex i becomes perm[i]
    out = np.empty_like(par)
    out[:, perm] = inv[par]
    roots, depth = fc.tree_roots(torch.from_numpy(out.astype(np.int32)).cuda())
    rr, rd = _ref(out) if T * n < 1 << 22 else (None, None)
    if rr is None:  # the defining equations, on the device
        p = torch.from_numpy(out).cuda()
        own = torch.arange(n, device="cuda").expand(T, n)
        top = p == n
        q = torch.where(top, own, p)
        assert torch.equal(roots.long(), torch.where(top, own, torch.gather(roots.long(), 1, q)))
        assert torch.equal(depth.long(), torch.where(top, 0, torch.gather(depth.long(), 1, q) + 1))
    else:
        np.testing.assert_array_equal(roots.cpu().numpy(), rr)
        np.testing.assert_array_equal(depth.cpu().numpy(), rd)


def test_cycle_in_a_later_window_is_refused():
    n, T = 5000, 3500
    par = torch.full((T, n), n, dtype=torch.int32, device="cuda")
    fc.tree_roots(par)
    par[T - 1, :3] = torch.tensor([1, 2, 0], dtype=torch.int32, device="cuda")
    with pytest.raises(fc.FcError):
        fc.tree_roots(par)


@pytest.mark.parametrize("kind", ["ba", "grid_weighted", "batch", "rooted"])
def test_automatic_forest_equals_the_recorded_one(kind):
    """Also with parents taken along and with one of the two outputs alone."""
    if kind == "batch":
        graphs, alphas = synth.uneven_batch(7, 5, n_min=1, n_max=900)
        u, offs = synth.union(graphs)
        G = fc.Graph.batch(u, offs, alphas)
        n, rows = u.n, 9
    elif kind == "rooted":
        g = synth.barabasi_albert(3000, 3, 4)
        G = fc.Graph.rooted(g, int(np.argmax(g.degrees())))
        n, rows = g.n, 9
    else:
        g = synth.barabasi_albert(3001, 3, 4) if kind == "ba" else synth.perturbed_grid(50, 61, 3)
        G = fc.Graph.from_csr(g, [0.2, 20.0])
        n, rows = g.n, 18
    with G:
        G.set_kernel(2)
        ref = G.sample(5, 9, want_roots=True, with_C=False)
        assert G.last_kernel() != 5
        G.set_kernel(0)
        for parents in (False, True):
            out = G.sample(5, 9, want_roots=True, want_parents=parents, with_C=False)
            assert G.last_kernel() == 5
            assert torch.equal(out["R"], ref["R"])
            assert torch.equal(out["roots"], ref["roots"]) and torch.equal(out["depths"], ref["depths"])
        for key in ("roots", "depths"):
            one = torch.empty(rows, n, dtype=torch.int32, device="cuda")
            R = torch.zeros(ref["R"].numel(), dtype=torch.int32, device="cuda")
            ptr = one.data_ptr()
            st = fc.lib().fc_sample_usts_forest(G._h, 5, 9, 0, R.data_ptr(), None, None,
                                                ptr if key == "roots" else None, ptr if key == "depths" else None,
                                                None, 0, None, torch.cuda.current_stream().cuda_stream)
            assert st == 0
            assert torch.equal(one.view(-1), ref[key].reshape(-1)), key

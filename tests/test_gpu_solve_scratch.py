"""Device scratch of the many-column solver: bounded on dense graphs, given
back when an allocation fails, and halved columns where all do not fit.  The
calls run on a memory pool of the test's own, so its counters and its size
limit are theirs alone."""
import contextlib
import ctypes

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

fc = pytest.importorskip("paper_2101_06192_gb300.fc")

MB = 1 << 20
USED_NOW, USED_HIGH = 7, 8  # CU_MEMPOOL_ATTR_USED_MEM_CURRENT, _HIGH


class _Props(ctypes.Structure):  # CUmemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("loc_type", ctypes.c_int),
                ("loc_id", ctypes.c_int), ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


class _Pool:
    def __init__(self, drv, handle):
        self.drv, self.handle = drv, handle

    def used(self, attr):
        torch.cuda.synchronize()
        v = ctypes.c_uint64()
        assert self.drv.cuMemPoolGetAttribute(self.handle, attr, ctypes.byref(v)) == 0
        return v.value


@contextlib.contextmanager
def _own_pool(max_size=0):
    drv = ctypes.CDLL("libcuda.so.1")
    dev, old, pool = torch.cuda.current_device(), ctypes.c_void_p(), ctypes.c_void_p()
    torch.cuda.synchronize()
    props = _Props(alloc_type=1, loc_type=1, loc_id=dev, max_size=max_size)
    assert drv.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) == 0
    assert drv.cuDeviceGetMemPool(ctypes.byref(old), dev) == 0
    assert drv.cuDeviceSetMemPool(dev, pool) == 0
    try:
        yield _Pool(drv, pool)
    finally:
        torch.cuda.synchronize()
        assert drv.cuDeviceSetMemPool(dev, old) == 0
        assert drv.cuMemPoolDestroy(pool) == 0


def _unit_columns(n, k):
    b = torch.zeros(k, n, dtype=torch.float64, device="cuda")
    b[torch.arange(k, device="cuda"), torch.arange(k, device="cuda") * (n // k)] = 1.0
    return b


def test_dense_graph_partial_sums_are_bounded():
    """Complete graph, 1024 columns: vectors 123 MB; segments of 128 entries
    would take 590 MB of partial sums.  L = n I - J: x = (b + alpha sum(b)) /
    (1 + alpha n) exactly."""
    n, k, alpha = 3000, 1024, 0.01
    with fc.Graph.from_csr(synth.complete(n), [alpha]) as G:
        b = _unit_columns(n, k)
        with _own_pool() as pool:
            x, _ = G.solve(b, rel_tol=1e-12)
            high = pool.used(USED_HIGH)
            assert pool.used(USED_NOW) == 0
    assert high < 450 * MB, high / MB
    ref = (b + alpha * b.sum(1, keepdim=True)) / (1.0 + alpha * n)
    # residual bound: |x - ref|_2 <= rel_tol |b|_2 / lambda_min, lambda_min = 1
    assert float((x - ref).norm(dim=1).max()) <= 1e-12


def test_group_on_dense_graph_is_bounded():
    """n = 2000, all columns in one batch: two matrices and the unit columns of
    32 MB each, vectors 160 MB; 512 MB of partial sums by segments of 128."""
    n, alpha = 2000, 0.5
    with fc.Graph.from_csr(synth.complete(n), [alpha]) as G:
        with _own_pool() as pool:
            S, far = G.group_closeness(3)
            high = pool.used(USED_HIGH)
            assert pool.used(USED_NOW) == 0
    assert high < 550 * MB, high / MB
    assert len(set(S.cpu().tolist())) == 3
    # every vertex alike: the trace of the inverse of L* without any k vertices
    Ls = np.full((n + 1, n + 1), -alpha)
    Ls[n, :] = Ls[:, n] = -1.0
    Ls[np.arange(n), np.arange(n)] = 1.0 + alpha * (n - 1)
    Ls[n, n] = n
    ref = [np.trace(np.linalg.inv(Ls[k:, k:])) for k in (1, 2, 3)]
    np.testing.assert_allclose(far.cpu().numpy(), ref, rtol=1e-9)


def test_columns_in_halves_when_the_scratch_does_not_fit():
    """30 columns of 2^17 vertices want 157 MB; within 120 MB they are solved as
    two halves, to the same tolerance."""
    n, k = 1 << 17, 30
    with fc.Graph.from_csr(synth.torus(512, 256), [1.0]) as G:
        b = _unit_columns(n, k)
        whole, _ = G.solve(b, rel_tol=1e-12)
        with _own_pool(120 * MB) as pool:
            x, it = G.solve(b, rel_tol=1e-12)
            assert pool.used(USED_NOW) == 0
    assert it > 0
    # both within rel_tol |b| / lambda_min of the solution
    assert float((x - whole).norm(dim=1).max()) <= 2e-12


def test_refused_allocation_leaves_nothing_behind():
    """A pool too small for one column (84 MB; pools grow in steps of 32 MB):
    FC_ENOMEM, no memory held, x as it was, and the next call is whole again."""
    n = 1 << 21
    with fc.Graph.from_csr(synth.torus(2048, 1024), [1.0]) as G:
        b = _unit_columns(n, 4)
        x = torch.full_like(b, 0.25)
        with _own_pool(32 * MB) as pool:
            with pytest.raises(fc.FcError) as e:
                G.solve(b, x=x)
            assert e.value.status == fc.FC_ENOMEM
            assert pool.used(USED_NOW) == 0
        assert bool((x == 0.25).all())
        x, _ = G.solve(b, rel_tol=1e-10)
    np.testing.assert_allclose(x.sum(1).cpu().numpy(), 1.0, atol=1e-7)  # 1^T (I + L)^-1 = 1^T


def test_refused_allocation_is_the_error_of_its_own_call():
    """One column, refused; the next call of the thread launches and returns."""
    g = synth.torus(2048, 1024)
    with fc.Graph.from_csr(g, [1.0]) as G:
        b = _unit_columns(g.n, 1)
        with _own_pool(32 * MB):
            with pytest.raises(fc.FcError) as e:
                G.solve(b)
            assert e.value.status == fc.FC_ENOMEM
            with fc.Graph.from_csr(synth.path(10), [1.0]) as P:
                assert P.sample(1, 4)["R"].numel() == 10

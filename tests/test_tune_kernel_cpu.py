"""The shipped launch shapes belong to the edge-record kernel: the tuner gives
them to it alone and probes for the CSR-walk kernel (host logic, no GPU)."""
import pytest

tune = pytest.importorskip("paper_2101_06192_gb300.tune")


class _Graph:
    """The benchmark graph's sizes (BA n = 2^20, m = 8); records what it is given."""
    n, nnz, weighted, n_alpha = 1 << 20, 16775658, False, 1

    def __init__(self, kernel_pref):
        self.kernel_pref = kernel_pref
        self.shapes = []

    def set_shape(self, *shape):
        self.shapes.append(shape)

    def set_start_order(self, order):
        self.order = order

    def last_shape(self):
        return {}


@pytest.mark.parametrize("kernel_pref", [1, 2])
def test_shipped_shapes_go_to_the_edge_record_kernel(monkeypatch, tmp_path, kernel_pref):
    probes = []
    monkeypatch.setattr(tune, "_CACHE", str(tmp_path / "shapes.json"))
    monkeypatch.setattr(tune, "_load", lambda path=None: {} if path is None else tune_load(path))
    monkeypatch.setattr(tune, "_time", lambda G, seed, probe: probes.append(G.shapes[-1]) or 1.0)
    G = _Graph(kernel_pref)
    got = tune.autotune(G, 1024)
    if kernel_pref == 2:
        assert got["cached"] == "shipped" and not probes
    else:
        assert "cached" not in got and len(probes) == len(tune.ORDERS) + len(tune.CANDIDATES)


tune_load = tune._load

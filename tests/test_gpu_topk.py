"""top-k: the selection (k <= 3072) and the full sort give the order of a
stable sort of (value, id) -- ties by id, -0.0 = +0.0, NaN last -- on crowded
values, at the edges of a block's sort and of the selection's capacity."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

fc = pytest.importorskip("paper_2101_06192_gb300.fc")


def _ref(d, k):
    key = np.where(d == 0.0, 0.0, d)
    return np.lexsort((np.arange(d.size), key))[:k]  # NumPy sorts NaN last


@pytest.mark.parametrize("n", [1, 2, 31, 1000, 1024, 1025, 4096, 5000, 70001, 1 << 20])
@pytest.mark.parametrize("kind", ["uniform", "ties", "one_value", "special"])
def test_topk_order(n, kind):
    rng = np.random.default_rng(n)
    if kind == "uniform":
        d = rng.random(n)
    elif kind == "ties":
        d = rng.integers(0, 7, n) / 1024.0
    elif kind == "one_value":
        d = np.full(n, 0.25)
    else:
        d = rng.choice([0.0, -0.0, np.nan, np.inf, -np.inf, -1.5, 1e-310, 2.0], n)
    dev = torch.from_numpy(d).cuda()
    for k in sorted({1, min(10, n), min(100, n), min(1024, n), min(3072, n), min(3073, n), min(5000, n)}):
        got = fc.top_k(dev, k).cpu().numpy()
        np.testing.assert_array_equal(got, _ref(d, k), err_msg=f"k={k}")

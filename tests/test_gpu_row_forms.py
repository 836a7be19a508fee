"""Propagation and best-first scoring by row form: narrow and wide aligned
rows, rows of any alignment and length, every element type, both sides of the
widths where the form changes.  Integer rows with squared distances below
2^24: exact."""
import numpy as np
import pytest

import oracle

from test_gpu_parity import assert_lists_exact, dev, host, knng

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DT = {"f32": torch.float32, "f16": torch.float16, "u8": torch.uint8}


def _graph(X, k):
    """An unfinished graph: leaf lists of one division."""
    perm, off = oracle.partition(X, 3, 0, 64)
    return oracle.leaf_knn(X, perm, off, k)


@pytest.mark.parametrize("dtype,d,offset", [
    ("f32", 1, 0), ("f32", 37, 0), ("f32", 36, 0), ("f32", 36, 1), ("f32", 208, 0), ("f32", 212, 0), ("f32", 130, 0),
    ("f16", 37, 0), ("f16", 96, 0), ("f16", 512, 0), ("f16", 516, 0), ("f16", 96, 2),
    ("u8", 37, 0), ("u8", 64, 0), ("u8", 64, 1), ("u8", 128, 0), ("u8", 200, 0), ("u8", 300, 0),
])
def test_rows_exact(dtype, d, offset):
    n, k = 900, 12
    rng = np.random.default_rng(d)
    X = rng.integers(0, 120 if d > 250 else 200, size=(n, d)).astype(np.float32)
    buf = torch.zeros(n * d + offset, dtype=DT[dtype], device="cuda")
    buf[offset:] = dev(X).to(DT[dtype]).reshape(-1)
    Xd = buf[offset:].view(n, d)
    ids, dd = _graph(X, k)
    gi, gd = knng().knng_propagate(Xd, dev(ids), dev(dd))
    oi, od = oracle.propagate(X, ids, k)
    assert_lists_exact(host(gi), host(gd), oi, od)
    for budget in (k, 57, 300):
        gi, gd = knng().knng_propagate_best_first(Xd, dev(ids), budget)
        oi, od = oracle.propagate_best_first(X, ids, k, budget)
        assert_lists_exact(host(gi), host(gd), oi, od)


@pytest.mark.parametrize("k,budget", [(1, 1), (33, 512), (64, 100), (5, 31), (20, 33)])
def test_best_first_sizes_exact(k, budget):
    rng = np.random.default_rng(k)
    X = rng.integers(0, 6, size=(700, 9)).astype(np.float32)  # many equal distances
    perm, off = oracle.partition(X, 3, 0, 150)
    ids, _ = oracle.leaf_knn(X, perm, off, k)
    for dtype in (torch.float32, torch.uint8):
        gi, gd = knng().knng_propagate_best_first(dev(X).to(dtype), dev(ids), budget, rounds=2)
        i1, _ = oracle.propagate_best_first(X, ids, k, budget)
        oi, od = oracle.propagate_best_first(X, i1, k, budget)
        assert_lists_exact(host(gi), host(gd), oi, od)

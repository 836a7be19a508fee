"""Exact k-NN with the pairs filtered on the tensor cores: ragged sizes, every
element type, lists from one query to several row tiles, and the queries that
the filter hands back (long lists of equal rows, rows that are not finite).

The rows are integers that bfloat16 does not hold (up to ten bits) with every
squared distance below 2^24, so FP32 distances are exact and the lists must
equal the oracle's bit for bit: the filter may only drop rows that are not in
the answer."""
import numpy as np
import pytest

import oracle

from test_gpu_parity import assert_lists_exact, dev, host, knng

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(X, q, k, Xd=None):
    gi, gd = knng().knng_exact_knn(dev(X) if Xd is None else Xd, dev(q.astype(np.int32)), k)
    knng().knng_sync()
    oi, od = oracle.knn_exact(X, k, q)
    assert_lists_exact(host(gi), host(gd), oi, od)


def _clustered(n, d, top, seed):
    rng = np.random.default_rng(seed)
    C = rng.integers(0, top, size=(20, d))
    X = C[rng.integers(0, 20, size=n)] + rng.integers(-6, 7, size=(n, d))
    return np.clip(X, 0, top).astype(np.float32)


@pytest.mark.parametrize("n,d,nq,k", [
    (2048, 37, 1, 1),       # the smallest filtered set, one query
    (2049, 37, 129, 64),    # one row past a tile, two query tiles, the largest k
    (5000, 3, 300, 20),     # one K slice, mostly padding
    (40000, 40, 1000, 20),
    (3001, 200, 64, 10),    # queries resident, four K slices
    (2500, 300, 140, 33),   # queries streamed with the rows
    (2600, 961, 20, 5),
])
def test_lists_equal_oracle(n, d, nq, k):
    top = int(np.sqrt((1 << 24) / d)) - 1  # d * top^2 < 2^24
    X = _clustered(n, d, min(top, 600), n + d)
    q = np.random.default_rng(d).choice(n, size=nq, replace=False)
    _check(X, q, k)


@pytest.mark.parametrize("dtype", [torch.float16, torch.uint8])
def test_element_types(dtype):
    X = _clustered(4000, 60, 255 if dtype == torch.uint8 else 500, 3)
    q = np.arange(0, 4000, 31)
    _check(X, q, 15, dev(X).to(dtype))


def test_more_queries_than_a_batch():
    X = _clustered(17000, 4, 600, 9)
    q = np.arange(17000)
    gi, gd = knng().knng_exact_knn(dev(X), dev(q.astype(np.int32)), 6)
    rows = np.r_[0:200, 16300:16500, 16900:17000]
    oi, od = oracle.knn_exact(X, 6, rows)
    assert_lists_exact(host(gi)[rows], host(gd)[rows], oi, od)


def test_long_lists_of_equal_rows_and_rows_not_finite():
    X = _clustered(6000, 24, 500, 4)
    X[1000:2500] = X[7]  # 1,500 equal rows: their lists overflow
    q = np.r_[0:40, 1000:1010, 2499, 5999]
    _check(X, q, 12)
    # infinite distances order after all others (the oracle's FP64 distance
    # of a finite row to these is infinite too)
    X[3000, 5] = np.inf
    q = q[q != 3000]
    _check(X, q, 12)


def test_queries_out_of_range_get_empty_rows():
    X = _clustered(3000, 16, 500, 6)
    q = np.array([5, -1, 3000, 2999, 7], dtype=np.int32)
    gi, gd = knng().knng_exact_knn(dev(X), dev(q), 4)
    gi, gd = host(gi), host(gd)
    assert (gi[1:3] == -1).all() and np.isinf(gd[1:3]).all()
    ok = np.array([0, 3, 4])
    oi, od = oracle.knn_exact(X, 4, q[ok])
    assert_lists_exact(gi[ok], gd[ok], oi, od)


def test_far_from_the_origin_and_captured_streams():
    # offset far above the spread: the bounds hold no row back and the
    # queries go to the direct form; a captured call takes it at once
    rng = np.random.default_rng(8)
    X = (1000 + rng.integers(0, 20, size=(5000, 30))).astype(np.float32)
    q = np.arange(0, 5000, 199)
    _check(X, q, 9)
    Xd, qd = dev(X), dev(q.astype(np.int32))
    ids = torch.empty(len(q), 9, dtype=torch.int32, device="cuda")
    dd = torch.empty(len(q), 9, dtype=torch.float32, device="cuda")
    knng().knng_exact_knn(Xd, qd, 9, ids=ids, dists=dd)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        knng().knng_exact_knn(Xd, qd, 9, ids=ids, dists=dd)
    ids.zero_()
    graph.replay()
    oi, od = oracle.knn_exact(X, 9, q)
    assert_lists_exact(host(ids), host(dd), oi, od)

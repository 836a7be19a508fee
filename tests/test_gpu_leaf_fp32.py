"""FP32 candidate stage and its selection at the sizes where they branch:
columns per lane 1 to 16, leaves that end inside a lane's columns, k' within
one lane minimum each (32) and beyond, ties at the cut, row blocks with a
single row, every element type and unaligned rows; k' above the staged limit.

Integer rows with squared distances below 2^24: candidate and FP32 distances
are exact, so the lists equal the oracle's bit for bit."""
import numpy as np
import pytest

import oracle

from test_gpu_parity import assert_lists_exact, dev, host, knng

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(X, Xd, T, g, k, mult=2, h=None):
    perm = knng().knng_partition(Xd, T, g, 3, h=h)
    ids, dd = knng().knng_leaf_knn(Xd, T, g, perm, k, 0, mult, h=h)
    off = knng().knng_leaf_offsets(X.shape[0], g)
    for t in range(T):
        oi, od = oracle.leaf_knn(X, host(perm)[t], off, k)
        assert_lists_exact(host(ids)[t], host(dd)[t], oi, od)


@pytest.mark.parametrize("n,d,k,g,top", [
    (1000, 40, 5, 32, 200), (1000, 33, 10, 44, 200), (900, 128, 10, 64, 200), (2000, 96, 20, 128, 200),
    (1537, 31, 20, 192, 200), (2000, 64, 20, 256, 200), (2049, 3, 20, 256, 9), (3000, 130, 20, 384, 200),
    (2000, 960, 10, 512, 100), (514, 8, 20, 257, 3), (64, 20, 20, 64, 200), (700, 5, 1, 4, 50),
])
def test_sizes_exact(n, d, k, g, top):
    X = np.random.default_rng(n + d).integers(0, top, size=(n, d)).astype(np.float32)
    _check(X, dev(X), 2, g, k)


@pytest.mark.parametrize("dtype", [torch.float16, torch.uint8])
def test_element_types_exact(dtype):
    X = np.random.default_rng(4).integers(0, 255, size=(1500, 50)).astype(np.float32)
    _check(X, dev(X).to(dtype), 2, 200, 16)


def test_unaligned_rows_exact():
    X = np.random.default_rng(5).integers(0, 255, size=(1500, 53)).astype(np.float32)
    buf = torch.zeros(1500 * 53 + 1, device="cuda")
    buf[1:] = dev(X).reshape(-1)
    _check(X, buf[1:].view(1500, 53), 2, 128, 12)


@pytest.mark.parametrize("k,mult", [(20, 2), (30, 2)])
def test_leaf_stage_is_the_first_call_of_a_handle(k, mult):
    X = np.random.default_rng(6).integers(0, 255, size=(1500, 50)).astype(np.float32)
    Xd = dev(X)
    perm = knng().knng_partition(Xd, 1, 128, 3)
    ids, dd = knng().knng_leaf_knn(Xd, 1, 128, perm, k, 0, mult, h=knng().Handle(0))
    oi, od = oracle.leaf_knn(X, host(perm)[0], knng().knng_leaf_offsets(1500, 128), k)
    assert_lists_exact(host(ids)[0], host(dd)[0], oi, od)

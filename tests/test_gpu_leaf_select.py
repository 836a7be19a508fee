"""Candidate selection and staged FP32 rescoring of the tensor-core leaf
kernel at the sizes where they branch: k' below, at and above the register
network's 32 and the row-per-thread limit of 48, leaves with a few points
more than k', ties at the cut, leaves of more than 256 points (three slices in
flight), every element type, rows that are not 16-byte aligned.

The rows hold multiples of 1/2 of magnitude < 64: exact in bfloat16 (so the
candidate distances and the FP32 distances are exact and the answer is the
exact leaf graph, with no tolerance), but not integers, so no leaf takes the
exact-leaf shortcut.  Few distinct values per entry at small d give many equal
distances."""
import numpy as np
import pytest

import oracle

from test_gpu_parity import assert_lists_exact, dev, host, knng

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("n,d,k,g,levels", [
    (3000, 96, 16, 200, 64),    # k' = 32: cut by the register network
    (3000, 40, 20, 256, 64),    # k' = 40
    (2500, 33, 20, 500, 64),    # k' = 40, leaves over 256 points, ragged d
    (4000, 3, 16, 128, 8),      # ties everywhere
    (1200, 64, 24, 256, 64),    # k' = 48: the row-per-thread limit, rescored in the kernel
    (1200, 64, 30, 256, 64),    # k' = 60: warp per row
    (900, 64, 10, 22, 64),      # leaves of 14 or 15 points: fewer members than k'
    (2000, 960, 10, 512, 64),   # rows in point order, 30 slices
])
def test_half_integer_rows_exact(dtype, n, d, k, g, levels):
    rng = np.random.default_rng(n + d + k)
    X = (0.5 + rng.integers(0, levels, size=(n, d)) * 0.5).astype(np.float32)
    Xd = dev(X) if dtype == "f32" else dev(X).half()
    T = 2
    perm = knng().knng_partition(Xd, T, g, 3)
    ids, dd = knng().knng_leaf_knn(Xd, T, g, perm, k, 1, 2)
    off = knng().knng_leaf_offsets(n, g)
    for t in range(T):
        oi, od = oracle.leaf_knn(X, host(perm)[t], off, k)
        assert_lists_exact(host(ids)[t], host(dd)[t], oi, od)


@pytest.mark.parametrize("ld,first", [(37, 0), (40, 1), (41, 2)])
def test_unaligned_rows_exact(ld, first):
    rng = np.random.default_rng(ld)
    n, d, k, g, T = 2000, 36, 12, 128, 2
    buf = torch.from_numpy((0.5 + rng.integers(0, 64, size=n * ld + 4) * 0.5).astype(np.float32)).cuda()
    Xd = buf[first:first + n * ld].view(n, ld)[:, :d]
    perm = knng().knng_partition(Xd, T, g, 3)
    ids, dd = knng().knng_leaf_knn(Xd, T, g, perm, k, 1, 2)
    off = knng().knng_leaf_offsets(n, g)
    for t in range(T):
        oi, od = oracle.leaf_knn(np.ascontiguousarray(host(Xd)), host(perm)[t], off, k)
        assert_lists_exact(host(ids)[t], host(dd)[t], oi, od)


def test_outlying_list_is_cut_by_a_warp():
    # one row's neighbours all lie in the columns of one thread: a list of
    # more than 32 candidates beside a short one
    n, d, k, g, T = 256, 64, 20, 256, 1
    rng = np.random.default_rng(5)
    X = (32.5 + rng.integers(0, 60, size=(n, d)) * 0.5).astype(np.float32)
    near = np.arange(28)  # columns of the half-0 thread
    X[near] = (0.5 + rng.integers(0, 8, size=(len(near), d)) * 0.5).astype(np.float32)
    Xd = dev(X)
    perm = knng().knng_partition(Xd, T, g, 3)
    ids, dd = knng().knng_leaf_knn(Xd, T, g, perm, k, 1, 2)
    oi, od = oracle.leaf_knn(X, host(perm)[0], knng().knng_leaf_offsets(n, g), k)
    assert_lists_exact(host(ids)[0], host(dd)[0], oi, od)

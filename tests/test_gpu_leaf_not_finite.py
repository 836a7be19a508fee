"""Leaf lists of finite rows beside rows that are not finite (infinite or NaN
entries): the others' lists are those of a set in which these rows lie far
away, for every candidate stage and selection branch.  A row block's last rows
belong to no row of the leaf and hold the next leaf's rows, infinite ones
among them."""
import numpy as np
import pytest

import oracle

from test_gpu_parity import dev, host, knng

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
@pytest.mark.parametrize("g,k", [(64, 5), (100, 20), (256, 24), (500, 12), (200, 40)])
def test_finite_rows_keep_their_lists(precision, dtype, g, k):
    rng = np.random.default_rng(g + k)
    n, d = 3000, 24
    X = rng.integers(-20, 21, size=(n, d)).astype(np.float32) + 0.5
    bad = rng.choice(n, size=60, replace=False)
    far = X.copy()
    far[bad] = 30000.0 + np.arange(60)[:, None]
    X[bad[:20], 3], X[bad[20:40], 5], X[bad[40:], 7] = np.inf, -np.inf, np.nan
    perm = np.arange(n, dtype=np.int32)
    ids, dd = knng().knng_leaf_knn(dev(X).to(dtype), 1, g, dev(perm[None]), k, precision, 2)
    knng().knng_sync()
    ids, dd = host(ids)[0], host(dd)[0]
    oi, od = oracle.leaf_knn(far, perm, knng().knng_leaf_offsets(n, g), k)
    ok = np.setdiff1d(np.arange(n), bad)
    if precision == 2:  # (E4M3 candidates of these rows are not exact)
        assert not np.isin(ids[ok], bad).any() and np.isfinite(dd[ok]).all()
    else:
        np.testing.assert_array_equal(dd[ok], od[ok])
        np.testing.assert_array_equal(ids[ok], oi[ok])

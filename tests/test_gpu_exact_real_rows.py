"""Exact k-NN of real-valued rows: the form that filters the pairs on the
tensor cores against the direct form (the one a captured call takes), bit for
bit.  The rows are not exact in bfloat16 and their distances are rounded, so
every margin of the filter's bound counts: few and many entries, unit rows,
rows of very different lengths, distances that agree to rounding around rank
k, and magnitudes down to where squares of the entries are subnormal."""
import numpy as np
import pytest

from test_gpu_parity import dev, host, knng

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def both_forms(X, q, k):
    """Lists of the filtered and of the direct form."""
    Xd, qd = dev(X), dev(q.astype(np.int32))
    gi, gd = knng().knng_exact_knn(Xd, qd, k)
    ids = torch.empty(len(q), k, dtype=torch.int32, device="cuda")
    dd = torch.empty(len(q), k, dtype=torch.float32, device="cuda")
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        knng().knng_exact_knn(Xd, qd, k, ids=ids, dists=dd)
    graph.replay()
    torch.cuda.synchronize()
    return (host(gi), host(gd)), (host(ids), host(dd))


def check(X, q, k):
    (gi, gd), (di, dd) = both_forms(X, q, k)
    np.testing.assert_array_equal(gd, dd)
    np.testing.assert_array_equal(gi, di)


def _rows(kind, n, d, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, d))
    if kind == "unit":
        X = np.abs(X) + 0.5
        X /= np.linalg.norm(X, axis=1, keepdims=True)
    elif kind == "lengths":
        X *= 10.0 ** rng.uniform(-2, 2, size=(n, 1))
    elif kind == "shells":
        # clusters whose rows lie at nearly one distance from the centre
        C = rng.standard_normal((n // 100 + 1, d))
        X = C[rng.integers(0, len(C), size=n)] + X / np.linalg.norm(X, axis=1, keepdims=True) * (
            1e-2 * (1.0 + 1e-6 * rng.standard_normal((n, 1))))
    return X.astype(np.float32)


@pytest.mark.parametrize("kind,n,d,nq,k", [
    ("normal", 2048, 1, 200, 10), ("normal", 4000, 3, 500, 20), ("normal", 3000, 64, 300, 64),
    ("unit", 4000, 960, 200, 10), ("unit", 2500, 1201, 130, 5), ("lengths", 5000, 48, 400, 16),
    ("shells", 6000, 32, 400, 30), ("shells", 4000, 200, 300, 12),
])
def test_filtered_lists_equal_direct_lists(kind, n, d, nq, k):
    X = _rows(kind, n, d, n + d)
    check(X, np.random.default_rng(d).choice(n, size=nq, replace=False), k)


@pytest.mark.parametrize("scale", [1e-15, 1e-18, 1e-20, 3e-21, 1e-21, 3e-22, 1e-22, 1e-23])
@pytest.mark.parametrize("d", [3, 8, 64])
def test_rows_of_very_small_magnitude(d, scale):
    # below about 1e-19 the squares of the entries (and of their rounding
    # errors long before) are subnormal: relative error terms alone do not
    # bound what they lose
    X = (np.random.default_rng(d).standard_normal((2048, d)) * scale).astype(np.float32)
    check(X, np.arange(0, 2048, 7), 10)


@pytest.mark.parametrize("count", [1, 2, 63, 64, 65, 300])
@pytest.mark.parametrize("kind", ["long", "not finite", "inexact", "long and not finite"])
def test_rows_far_above_the_others(kind, count):
    # up to 64 such rows are taken out of the bounds and listed for every
    # query, more loosen the bounds (long rows, rows bfloat16 does not hold)
    # or send all queries to the direct form (rows that are not finite).  The
    # far rows are near one another, and some are queries.
    rng = np.random.default_rng(count)
    n, d = 4000, 24
    X = rng.integers(-100, 101, size=(n, d)).astype(np.float32)
    far = rng.choice(n, size=count, replace=False)
    if kind != "not finite":
        X[far] = (37.3 + rng.standard_normal((count, d))) * (1.0 if kind == "inexact" else 5000.0)
    if kind in ("not finite", "long and not finite"):
        for i in far[::2] if kind == "long and not finite" else far:
            X[i, rng.integers(d)] = (np.inf, -np.inf, np.nan, 3e38)[rng.integers(4)]
    q = np.unique(np.r_[rng.choice(n, size=150), far[:20]])
    check(X, q, 15)

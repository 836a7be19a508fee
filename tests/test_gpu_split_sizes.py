"""Median splits on the 32-bit keys with ties in position order: block sizes
by node size (up to 1,024, 2,048, 8,192 points and the multi-block split), all
keys equal, two keys, a few keys, negative and positive keys, several levels
of directions per launch.  The leaf sets must equal the oracle's."""
import numpy as np
import pytest

import oracle

from test_gpu_parity import dev, host, knng

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 257, 1024, 1025, 2049, 4100, 8192, 8193, 16385, 40000])
@pytest.mark.parametrize("kind", ["equal", "two", "few", "normal"])
def test_leaf_sets_equal_oracle(n, kind):
    rng = np.random.default_rng(n)
    d = 5
    if kind == "equal":
        X = np.full((n, d), 1.5, dtype=np.float32)
    elif kind == "two":
        X = np.where(rng.random((n, 1)) < 0.3, -2.25, 3.5).astype(np.float32) * np.ones((1, d), np.float32)
    elif kind == "few":
        X = rng.integers(-2, 3, size=(n, 1)).astype(np.float32) * np.arange(1, d + 1, dtype=np.float32) + 0.25
    else:
        X = rng.normal(size=(n, d)).astype(np.float32)
    g = 2 if n < 1000 else 100
    T = 2
    perm = host(knng().knng_partition(dev(X), T, g, 11))
    for t in range(T):
        want, _ = oracle.partition(X, 11, t, g)
        np.testing.assert_array_equal(perm[t], want)


def test_directions_of_a_run_of_levels():
    # wide rows: the directions of all levels exceed one launch's 64 MB
    rng = np.random.default_rng(1)
    X = rng.normal(size=(9000, 4000)).astype(np.float32)
    perm = host(knng().knng_partition(dev(X), 1, 4, 5))
    want, _ = oracle.partition(X, 5, 0, 4)
    np.testing.assert_array_equal(perm[0], want)

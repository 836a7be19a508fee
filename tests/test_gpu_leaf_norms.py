"""Squared norms in the FP32 leaf candidate stage: a zero row's candidate
distances are the others' norms alone (every product is 0), so with k' = k
its list shows how the stage's norms rank.  Norms a few rounding errors apart
must be ranked against FP64 as well as by a sum over 32 lanes (fixed partial
sums and five pairwise rounds, restated here in NumPy); one chain of d
additions misses two to fifteen times as many."""
import numpy as np
import pytest

from test_gpu_parity import dev, host, knng

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _lane_norms(X):
    n, d = X.shape
    Z = np.zeros((n, -(-d // 128) * 128), np.float32)
    Z[:, :d] = X
    p = np.zeros((n, 32), np.float32)
    for c in range(0, Z.shape[1], 128):
        for e in range(4):  # (the FP64 sum of an exact product rounds once: an FMA)
            v = Z[:, c + e:c + 128:4].astype(np.float64)
            p = (v * v + p).astype(np.float32)
    for o in (16, 8, 4, 2, 1):
        p = p + p[:, np.arange(32) ^ o]
    return p[:, 0]


def _misses(lists, nearest):
    return sum(len(set(a) - set(b)) for a, b in zip(lists, nearest))


@pytest.mark.parametrize("n,g,d", [(8000, 64, 2048), (20000, 200, 960), (60000, 256, 128), (64000, 500, 300)])
def test_norms_rank_no_worse_than_lane_sums(n, g, d):
    k = 10
    rng = np.random.default_rng(d)
    X = rng.standard_normal((n, d))
    X /= np.linalg.norm(X, axis=1, keepdims=True)
    off = np.asarray(knng().knng_leaf_offsets(n, g))
    spread = 2e-7 * np.diff(off).max()
    X = (X * np.sqrt(1.0 + spread * rng.random((n, 1)))).astype(np.float32)
    X[off[:-1]] = 0.0
    exact, lane = (X.astype(np.float64) ** 2).sum(1), _lane_norms(X)
    nearest, by_lane = [], []
    for b, e in zip(off[:-1], off[1:]):
        nearest.append(b + 1 + np.argsort(exact[b + 1:e], kind="stable")[:k])
        by_lane.append(b + 1 + np.argsort(lane[b + 1:e], kind="stable")[:k])
    perm = torch.arange(n, dtype=torch.int32, device="cuda").reshape(1, n)
    ids, _ = knng().knng_leaf_knn(dev(X), 1, g, perm, k, knng().PREC_FP32, 1)
    got = host(ids)[0][off[:-1]]
    # (counts of rare events: three standard deviations)
    lanes = _misses(by_lane, nearest)
    assert _misses(got, nearest) <= lanes + 3.0 * np.sqrt(max(lanes, 4))

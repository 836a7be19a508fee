"""Loss and gradient of the split-feature network at the sizes where the tiled
kernels can go wrong: ragged tiles in every dimension, batches shorter than
one slice or row block, both output widths.  Reference: the FP64 oracle.

Tolerance: every product is FP32 and the longest chain of additions is one
slice of the batch (at most a few hundred terms) plus the slices, so a
block's error is below 1e-4 of its norm even with the cancellation of the
centred statistics; 1e-3 is the bound of the network's other gradient test."""
import numpy as np
import pytest

from oracle import mlp as omlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,H,C,B", [(1, 16, 16, 2), (37, 48, 32, 65), (96, 256, 16, 1000), (130, 80, 16, 193),
                                     (64, 64, 32, 2049), (257, 240, 32, 33)])
def test_gradient_sizes(d, H, C, B):
    import paper_1307_7852_gb300 as k
    net = k.Mlp(d, H, C, seed=d + B)
    rng = np.random.default_rng(B)
    Xi = rng.normal(size=(B, d)).astype(np.float32)
    Xp = np.concatenate([Xi, (Xi + 0.3 * rng.normal(size=(B, d))).astype(np.float32)])
    loss, g = net.loss_grad(torch.from_numpy(Xp).cuda())
    L, parts = omlp.loss_and_grads(Xp, *net.get_params(), lam=0.05, eps=1e-4)
    assert abs(loss - L) <= 1e-4 * abs(L)
    g = g.cpu().numpy().astype(np.float64)
    total = np.sqrt(sum(np.sum(p ** 2) for p in parts))
    o = 0
    for p in parts:
        err = np.linalg.norm(g[o:o + p.size] - p.ravel())
        assert err <= 1e-3 * np.linalg.norm(p) + 1e-5 * total
        o += p.size

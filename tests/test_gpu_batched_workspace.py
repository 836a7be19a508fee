"""A recorded batched build after another call has grown, and so moved, the
handle's workspace: the graph holds addresses in the old one and must be
recorded again."""
import numpy as np
import pytest

from paper_1307_7852_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_replay_after_the_workspace_moved():
    import paper_1307_7852_gb300 as knng
    Xs = [torch.from_numpy(synthetic.gaussian_mixture(n, 24, centers=6, std=0.2, seed=n)).cuda() for n in (700, 3000, 90)]
    k, T, g, R, seed = 6, 3, 40, 1, 11
    outs = [(torch.empty(len(X), k, dtype=torch.int32, device="cuda"),
             torch.empty(len(X), k, dtype=torch.float32, device="cuda")) for X in Xs]
    h = knng.Handle(0)
    ref = [knng.knng_build(X, k, T, g, R, seed) for X in Xs]
    for n in (20_000, 150_000):
        knng.knng_build_batched(Xs, k, T, g, R, seed, outs=outs, h=h)
        big = torch.randn(n, 40, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
        knng.knng_build(big, 10, 4, 64, 1, seed, h=h)  # grows the workspace
        for i, d in outs:
            i.zero_()
            d.zero_()
        knng.knng_build_batched(Xs, k, T, g, R, seed, outs=outs, h=h)
        torch.cuda.synchronize()
        for (ri, rd), (gi, gd) in zip(ref, outs):
            np.testing.assert_array_equal(gi.cpu().numpy(), ri.cpu().numpy())
            np.testing.assert_array_equal(gd.cpu().numpy(), rd.cpu().numpy())
    knng.knng_sync(h)

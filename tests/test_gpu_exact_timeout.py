"""Bounded waits of the exact k-NN call's tensor-core passes: with a limit of a
few cycles its waits give up on copies and MMAs that are still in flight.
Every CTA then waits for them under the one-second limit before it frees its
tensor memory and returns, knng_sync reports KNNG_ERR_TIMEOUT, the lists come
from the direct form, and the same handle works once the default limit is
back.  One tile of one K slice per CTA (every copy is issued before the first
wait runs out), several tiles with resident queries, and streamed queries."""
import numpy as np
import pytest

import oracle

from test_gpu_exact_filter import _clustered
from test_gpu_parity import assert_lists_exact, dev, host, knng

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KNNG_ERR_TIMEOUT = -5


@pytest.mark.parametrize("n,d,nq", [(2048, 40, 10), (30000, 130, 700), (6000, 300, 300)])
def test_waits_run_out_and_the_lists_stay_right(n, d, nq):
    k = knng()
    X = _clustered(n, d, min(int(np.sqrt((1 << 24) / d)) - 1, 600), n + d)
    q = np.random.default_rng(d).choice(n, size=nq, replace=False).astype(np.int32)
    oi, od = oracle.knn_exact(X, 9, q)
    Xd, qd = dev(X), dev(q)
    h = k.Handle(0)
    k.knng_set_wait_limit(8, h)
    gi, gd = k.knng_exact_knn(Xd, qd, 9, h=h)
    with pytest.raises(k.KnngError) as e:
        k.knng_sync(h)
    assert e.value.code == KNNG_ERR_TIMEOUT
    assert_lists_exact(host(gi), host(gd), oi, od)
    k.knng_set_wait_limit(0, h)
    gi, gd = k.knng_exact_knn(Xd, qd, 9, h=h)
    k.knng_sync(h)
    assert_lists_exact(host(gi), host(gd), oi, od)


def test_an_earlier_calls_timeout_leaves_the_filter_on():
    # the handle's error word stays set until knng_sync reads it
    from test_gpu_exact_cost import best_ms, call_and_direct, normal_rows
    k = knng()
    X = normal_rows(60000, 64, 5)
    q = torch.arange(1000, dtype=torch.int32, device="cuda") * 60
    direct = call_and_direct(X, q, 10)[1]
    h = k.Handle(0)
    perm = k.knng_partition(X, 1, 128, 3, h=h)
    k.knng_sync(h)
    k.knng_set_wait_limit(8, h)
    k.knng_leaf_knn(X, 1, 128, perm, 10, k.PREC_BF16, 2, h=h)
    k.knng_set_wait_limit(0, h)
    assert best_ms(lambda: k.knng_exact_knn(X, q, 10, h=h)) < 0.5 * direct
    with pytest.raises(k.KnngError):
        k.knng_sync(h)

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

"""What the exact k-NN call costs on sets whose rows its filter cannot tell
apart or cannot bound: little more than the direct form, which then answers."""
import pytest

from test_gpu_parity import knng

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def best_ms(f, reps=6):
    f()
    out = []
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        b.synchronize()
        out.append(a.elapsed_time(b))
    return min(out)


def call_and_direct(X, q, k):
    """Best times of the call and of the direct form (a captured call)."""
    ids = torch.empty(len(q), k, dtype=torch.int32, device="cuda")
    dd = torch.empty(len(q), k, dtype=torch.float32, device="cuda")
    knng().knng_exact_knn(X, q, k, ids=ids, dists=dd)  # (the handle exists before the capture)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        knng().knng_exact_knn(X, q, k, ids=ids, dists=dd)
    return best_ms(lambda: knng().knng_exact_knn(X, q, k, ids=ids, dists=dd)), best_ms(graph.replay)


def normal_rows(n, d, seed):
    return torch.randn(n, d, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda")


@pytest.mark.parametrize("kind", ["equal", "not finite"])
def test_handed_back_sets_cost_the_direct_form(kind):
    # before: one atomic per pair, 8 to 11 % of the direct form (equal rows),
    # and both passes over rows that no bound holds for
    n, nq = 60000, 2000
    X = normal_rows(n, 64, 1)
    if kind == "equal":
        X[:] = X[0].clone()
    else:
        X[::2, 1] = float("nan")  # (far more rows than can be taken out)
    q = torch.arange(nq, dtype=torch.int32, device="cuda") * (n // nq)
    call, direct = call_and_direct(X, q, 10)
    assert call < 1.05 * direct


@pytest.mark.parametrize("kind", ["one long row", "one infinite row"])
def test_one_odd_row_leaves_the_filter_to_the_others(kind):
    # the bound of every query took its margins from the largest row: all
    # queries went to the direct form
    n, nq = 60000, 2000
    X = normal_rows(n, 64, 2)
    X[n // 2] = X[n // 2] * 300.0 if kind == "one long row" else float("inf")
    q = torch.arange(nq, dtype=torch.int32, device="cuda") * (n // nq) + 1
    call, direct = call_and_direct(X, q, 10)
    assert call < 0.5 * direct

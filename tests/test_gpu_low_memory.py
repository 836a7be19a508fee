"""Calls with too little device memory for their usual scratch: they take the
forms that need less (a leaf stage that needed none before its candidates
were staged through memory still runs), and the scratch that knng_exact_knn
keeps is given back to a build that needs the room.  The rows hold small
integers, so every form's distances and candidates are exact and the lists
must be the same."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
MB = 1 << 20


def _rows(n, d, dtype=torch.float32):
    gen = torch.Generator(device="cuda").manual_seed(n + d)
    return torch.randint(0, 200, (n, d), generator=gen, device="cuda").to(dtype)


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _workspace(call):
    """Bytes that call's workspace needs, without the room to grow; its result."""
    import paper_1307_7852_gb300 as knng
    h = knng.Handle(0)
    before = _free()
    out = call(h)
    used = before - _free()
    return int((used - MB) / 1.125), out


def _with_free(left, call):
    free = _free()
    filler = torch.empty(free - left, dtype=torch.uint8, device="cuda")
    try:
        torch.cuda.synchronize()
        return call()
    finally:
        torch.cuda.synchronize()
        del filler
        torch.cuda.empty_cache()


def _outputs(*shape):
    return (torch.zeros(*shape, dtype=torch.int32, device="cuda"), torch.zeros(*shape, device="cuda"))


def _same(a, b):
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x.cpu().numpy(), y.cpu().numpy())


@pytest.mark.parametrize("precision,dtype", [(0, torch.float32), (0, torch.uint8), (1, torch.uint8), (1, torch.float32)])
def test_leaf_stage_without_room_for_its_candidates(precision, dtype):
    import paper_1307_7852_gb300 as knng
    n, T, g, k = 300_000, 8, 100, 20
    X = _rows(n, 32, dtype)
    perm = torch.arange(n, dtype=torch.int32, device="cuda").repeat(T, 1)
    want, got = _outputs(T, n, k), _outputs(T, n, k)
    need, _ = _workspace(lambda h: knng.knng_leaf_knn(X, T, g, perm, k, precision, 2, ids=want[0], dists=want[1], h=h))
    cand = T * n * 2 * k * 2  # bytes of the staged candidates
    h = knng.Handle(0)
    knng.knng_leaf_knn(X[:1000], 1, g, perm[:1, :1000].contiguous(), k, precision, 2, h=h)  # (modules loaded)
    _with_free(need - cand // 2,
               lambda: knng.knng_leaf_knn(X, T, g, perm, k, precision, 2, ids=got[0], dists=got[1], h=h))
    _same(got, want)


def test_build_without_room_for_its_usual_scratch():
    import paper_1307_7852_gb300 as knng
    n, T, g, k = 300_000, 8, 100, 20
    X = _rows(n, 32)
    want, got = _outputs(n, k), _outputs(n, k)
    need, _ = _workspace(lambda h: knng.knng_build(X, k, T, g, 1, 3, 0, ids=want[0], dists=want[1], h=h))
    h = knng.Handle(0)
    _with_free(need - 40 * MB, lambda: knng.knng_build(X, k, T, g, 1, 3, 0, ids=got[0], dists=got[1], h=h))
    _same(got, want)


def test_exact_scratch_makes_room_for_a_build():
    import paper_1307_7852_gb300 as knng
    n, T, g, k = 300_000, 8, 100, 20
    X = _rows(n, 32)
    want, got, wide = _outputs(n, k), _outputs(n, k), _rows(400_000, 300)
    need, _ = _workspace(lambda h: knng.knng_build(X, k, T, g, 1, 3, 0, ids=want[0], dists=want[1], h=h))
    h = knng.Handle(0)
    q = torch.arange(0, 400_000, 1000, dtype=torch.int32, device="cuda")
    before = knng.knng_exact_knn(wide, q, 5, h=h)  # keeps over 300 MB
    _with_free(need - 100 * MB, lambda: knng.knng_build(X, k, T, g, 1, 3, 0, ids=got[0], dists=got[1], h=h))
    _same(got, want)
    _same(knng.knng_exact_knn(wide, q, 5, h=h), before)


def test_captured_leaf_stage_allocates_nothing():
    # a recording cannot grow the workspace: the stage takes the form that
    # fits what the handle has
    import paper_1307_7852_gb300 as knng
    n, T, g, k = 60_000, 2, 100, 20
    X = _rows(n, 32)
    perm = torch.arange(n, dtype=torch.int32, device="cuda").repeat(T, 1)
    want, got = _outputs(T, n, k), _outputs(T, n, k)
    knng.knng_leaf_knn(X, T, g, perm, k, 0, 2, ids=want[0], dists=want[1])
    h = knng.Handle(0)
    knng.knng_leaf_knn(X[:n // 2], 1, g, perm[:1, :n // 2].contiguous(), k, 0, 2, h=h)  # a workspace half as large
    knng.knng_partition(X, 1, g, 3, h=h)  # (the plan for n points)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        knng.knng_leaf_knn(X, T, g, perm, k, 0, 2, ids=got[0], dists=got[1], h=h)
    graph.replay()
    torch.cuda.synchronize()
    _same(got, want)

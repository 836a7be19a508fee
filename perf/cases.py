"""Workloads of the k-NN graph library, as its users run them.

Every case is one call (or one stage call) of the public Python entry points
on seeded synthetic points shaped like the library's target data: SIFT-like
byte values, GIST-like unit rows, Gaussian mixtures and unit-sphere mixtures.
The points are generated on the GPU from the seed alone.
"""
import math

import torch

import paper_1307_7852_gb300 as knng

DEVICE = "cuda:0"
PRECISION = {"fp32": knng.PREC_FP32, "bf16": knng.PREC_BF16, "fp8": knng.PREC_FP8E4M3}
PARTITIONER = {"random": knng.PART_RANDOM, "pca": knng.PART_PCA, "features": knng.PART_FEATURES}
METRIC = {"l2": knng.METRIC_L2, "cosine": knng.METRIC_COSINE}
ELEMENT = {"f32": torch.float32, "f16": torch.float16, "u8": torch.uint8}
ELEMENT_BYTES = {"f32": 4, "f16": 2, "u8": 1}
TREE_SEED = 7  # a program fixes its partition seed; the points change


def listed():
    return [
        # the smallest whole build: a small descriptor set, graph wanted at
        # once; latency and launches count
        dict(name="build_sift10k_fp32", op="build", data="sift", dtype="f32", n=10_000, d=128, centers=64, k=10, T=4,
             g=64, R=1, precision="fp32", metric="l2", partitioner="random"),
        # the headline: one million SIFT descriptors
        dict(name="build_sift1m_bf16", op="build", data="sift", dtype="f32", n=1_000_000, d=128, centers=1024, k=20,
             T=8, g=256, R=2, precision="bf16", metric="l2", partitioner="random"),
        # one million wide real-valued rows (GIST-960): the largest rows
        dict(name="build_gist1m_bf16", op="build", data="gist", dtype="f32", n=1_000_000, d=960, centers=256, k=10,
             T=8, g=512, R=1, precision="bf16", metric="l2", partitioner="random"),
        # 384-entry GIST rows, the FP8 candidate stage with k' = 40, a ragged
        # number of points and a leaf size that is no power of two
        dict(name="build_gist384_fp8", op="build", data="gist", dtype="f32", n=300_007, d=384, centers=256, k=20, T=6,
             g=500, R=1, precision="fp8", metric="l2", partitioner="random"),
        # cosine metric on principal-direction trees, rows of 200 entries
        dict(name="build_cosine_pca", op="build", data="mixture", dtype="f32", n=200_003, d=200, centers=256, k=16,
             T=5, g=200, R=1, precision="bf16", metric="cosine", partitioner="pca"),
        # many independent sets of uneven size in one recorded launch
        dict(name="batched256_bf16", op="batched", sets=256, n_lo=2_000, n_hi=200_000, k=10, T=6, g=128, R=1,
             precision="bf16"),
        # half-precision unit vectors, trees on the network's features
        dict(name="learned2m_f16", op="learned", data="sphere", dtype="f16", n=2_000_000, d=96, centers=4096, k=20,
             T=4, g=256, R=1, precision="bf16", hidden=256, outputs=16, partitioner="features"),
        # leaf graphs alone, FP32 candidate stage on real-valued rows
        dict(name="leaf_mix400k_fp32", op="leaf", data="mixture", dtype="f32", n=400_000, d=128, centers=256, k=20,
             T=4, g=256, precision="fp32"),
        # refining a given graph by propagation on real-valued rows
        dict(name="propagate_mix300k", op="propagate", data="mixture", dtype="f32", n=300_001, d=256, centers=256,
             k=20, T=2, g=128, R=2, scheme="first_order", budget=0),
        # budgeted best-first refinement on byte descriptors
        dict(name="best_first_u8", op="propagate", data="sift", dtype="u8", n=200_000, d=128, centers=256, k=16, T=2,
             g=128, R=1, scheme="best_first", budget=200),
        # exact lists of a 10,000-point sample: measuring a graph's recall
        dict(name="exact_sample10k", op="exact_knn", data="sift", dtype="f32", n=1_000_000, d=128, centers=1024,
             k=20, queries=10_000),
        # one training step's loss and gradient of the split-feature network
        dict(name="mlp_grad_b4096", op="mlp_grad", d=96, hidden=256, outputs=16, edges=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["build", "build", "build", "build", "batched", "learned", "leaf", "propagate", "propagate",
                     "exact_knn", "mlp_grad"])
    if op == "mlp_grad":
        return dict(op=op, d=rng.choice([32, 64, 96, 100, 128]), hidden=rng.choice([64, 128, 256]),
                    outputs=rng.choice([16, 32]), edges=_log_int(rng, 300, 8192))
    if op == "batched":
        return dict(op=op, sets=rng.randint(5, 64), n_lo=2_000, n_hi=_log_int(rng, 10_000, 200_000),
                    k=rng.randint(5, 16), T=rng.randint(2, 6), g=rng.choice([64, 100, 128]), R=rng.randint(0, 1),
                    precision=rng.choice(["bf16", "fp8", "fp32"]))
    if op == "learned":
        return dict(op=op, data="sphere", dtype=rng.choice(["f16", "f32"]), n=_log_int(rng, 20_000, 1_500_000),
                    d=rng.choice([64, 96, 128]), centers=1024, k=rng.randint(8, 20), T=rng.randint(2, 4),
                    g=rng.choice([128, 200, 256]), R=1, precision="bf16", hidden=rng.choice([64, 256]), outputs=16,
                    partitioner=rng.choice(["features", "random"]))
    data = rng.choice(["sift", "gist", "mixture"])
    d = {"sift": [64, 96, 100, 128], "gist": [384, 512, 960], "mixture": [37, 64, 128, 200, 256]}[data]
    d = rng.choice(d)
    dtype = rng.choice(["f32", "u8"]) if data == "sift" else rng.choice(["f32", "f32", "f16"])
    n_hi = 400_000 if d > 256 else 1_000_000
    if op == "exact_knn":
        return dict(op=op, data=data, dtype=dtype, n=_log_int(rng, 5_000, n_hi // 2), d=d, centers=256,
                    k=rng.randint(1, 50), queries=_log_int(rng, 10, 4_000))
    if op == "leaf":
        return dict(op=op, data=data, dtype=dtype, n=_log_int(rng, 5_000, n_hi // 4), d=d, centers=128,
                    k=rng.randint(5, 30), T=rng.randint(1, 4), g=rng.choice([64, 100, 200, 256, 400, 512]),
                    precision=rng.choice(["fp32", "bf16", "fp8"]))
    if op == "propagate":
        scheme = rng.choice(["first_order", "first_order", "best_first"])
        k = rng.randint(6, 32)
        return dict(op=op, data=data, dtype=dtype, n=_log_int(rng, 5_000, n_hi // 4), d=d, centers=128, k=k, T=2,
                    g=rng.choice([100, 128, 200]), R=rng.randint(1, 2), scheme=scheme,
                    budget=rng.randint(k, 300) if scheme == "best_first" else 0)
    g = rng.choice([64, 100, 128, 200, 256, 400, 512])
    return dict(op=op, data=data, dtype=dtype, n=_log_int(rng, 3_000, n_hi // 2), d=d, centers=256,
                k=rng.randint(5, min(32, g // 2 - 1)), T=rng.randint(2, 8), g=g, R=rng.randint(0, 2),
                precision=rng.choice(["bf16", "bf16", "fp8", "fp32"]), metric=rng.choice(["l2", "l2", "l2", "cosine"]),
                partitioner=rng.choice(["random", "random", "random", "pca"]))


# ----------------------------------------------------------------- inputs --
def _generator(seed, stream=0):
    return torch.Generator(device=DEVICE).manual_seed(1_000_003 * (seed + 1) + stream)


def _points(data, n, d, centers, dtype, gen):
    """n points of a Gaussian mixture of the named law, rows of d entries."""
    if data == "sift":
        C = torch.rand(centers, d, generator=gen, device=DEVICE) * 255.0
        std = 20.0
    elif data == "gist":
        C = torch.rand(centers, d, generator=gen, device=DEVICE)
        std = 0.1
    else:
        C = torch.randn(centers, d, generator=gen, device=DEVICE)
        std = 0.1
        if data == "sphere":
            C /= C.norm(dim=1, keepdim=True)
            std = 0.05
    X = torch.empty(n, d, dtype=ELEMENT[dtype], device=DEVICE)
    step = 1 << 18
    for s in range(0, n, step):
        m = min(step, n - s)
        lab = torch.randint(centers, (m,), generator=gen, device=DEVICE)
        v = C[lab] + std * torch.randn(m, d, generator=gen, device=DEVICE)
        if data == "sift":
            v = v.round_().clamp_(0.0, 255.0)
        elif data == "gist":
            v = v.clamp_(0.0, 1.0)
            v /= v.norm(dim=1, keepdim=True)
        elif data == "sphere":
            v /= v.norm(dim=1, keepdim=True)
        X[s:s + m] = v.to(X.dtype)
    return X


def _leaf_sizes(n, g):
    sizes = [n]
    while any(m > g for m in sizes):
        sizes = [h for m in sizes for h in ((m // 2, m - m // 2) if m > g else (m,))]
    return sizes


def _divisions(X, T, g, gen):
    """T random divisions of the points into leaves (perm [T, n] int32, ids
    ascending inside a leaf), the layout of knng_partition."""
    n, d = X.shape
    perm = torch.empty(T, n, dtype=torch.int32, device=DEVICE)
    for t in range(T):
        order = torch.arange(n, device=DEVICE)
        sizes = [n]
        while any(m > g for m in sizes):
            s = torch.empty(n, device=DEVICE)
            a = torch.randn(d, generator=gen, device=DEVICE)
            for i in range(0, n, 1 << 18):
                s[i:i + (1 << 18)] = X[i:i + (1 << 18)].float() @ a
            seg = torch.repeat_interleave(torch.arange(len(sizes), device=DEVICE),
                                          torch.tensor(sizes, device=DEVICE))
            by_value = torch.argsort(s[order], stable=True)
            order = order[by_value[torch.argsort(seg[by_value], stable=True)]]
            sizes = [h for m in sizes for h in ((m // 2, m - m // 2) if m > g else (m,))]
        seg = torch.repeat_interleave(torch.arange(len(sizes), device=DEVICE), torch.tensor(sizes, device=DEVICE))
        by_id = torch.argsort(order, stable=True)
        perm[t] = order[by_id[torch.argsort(seg[by_id], stable=True)]].to(torch.int32)
    return perm


def _leaf_lists(X, perm, g, k):
    """Brute-force lists inside every leaf in 64 bits: ids and squared
    distances, [T, n, k]."""
    T, n = perm.shape
    sizes = torch.tensor(_leaf_sizes(n, g), device=DEVICE)
    off = torch.cumsum(sizes, 0) - sizes
    mx = int(sizes.max())
    col = torch.arange(mx, device=DEVICE)
    ids = torch.empty(T, n, k, dtype=torch.int64, device=DEVICE)
    dist = torch.empty(T, n, k, dtype=torch.float64, device=DEVICE)
    step = max(1, (1 << 26) // (mx * max(mx, X.shape[1])))
    for t in range(T):
        for s in range(0, len(sizes), step):
            live = col[None, :] < sizes[s:s + step, None]
            pos = (off[s:s + step, None] + col[None, :]).clamp_(max=n - 1)
            mem = perm[t][pos].long()
            V = X[mem].double()
            q = (V * V).sum(2)
            D = (q[:, :, None] + q[:, None, :] - 2.0 * torch.bmm(V, V.transpose(1, 2))).clamp_(min=0.0)
            D.masked_fill_(~live[:, None, :], math.inf)
            D.diagonal(dim1=1, dim2=2).fill_(math.inf)
            dv, di = torch.topk(D, k, dim=2, largest=False, sorted=True)
            nb = torch.gather(mem[:, None, :].expand(-1, mx, -1), 2, di)
            ids[t, mem[live]] = nb[live]
            dist[t, mem[live]] = dv[live]
    return ids, dist


def _best(ids, dist, own, k):
    """The k nearest distinct ids of every row (own[row] excluded)."""
    ids, at = torch.sort(ids, dim=1)
    dist = torch.gather(dist, 1, at)
    bad = ids == own[:, None]
    bad[:, 1:] |= ids[:, 1:] == ids[:, :-1]
    dist = dist.masked_fill(bad, math.inf)
    dv, at = torch.sort(dist, dim=1, stable=True)
    return torch.gather(ids, 1, at[:, :k]), dv[:, :k]


def _given_graph(X, case, gen):
    """A graph to refine: the union of T divisions' leaf graphs."""
    k = case["k"]
    ids, dist = _leaf_lists(X, _divisions(X, case["T"], case["g"], gen), case["g"], k)
    n = X.shape[0]
    gi, gd = _best(ids.permute(1, 0, 2).reshape(n, -1), dist.permute(1, 0, 2).reshape(n, -1).float(),
                   torch.arange(n, device=DEVICE), k)
    return gi.to(torch.int32).contiguous(), gd.contiguous()


def _network(case, gen):
    d, H, C = case["d"], case["hidden"], case["outputs"]

    def normal(*shape, scale=1.0):
        return torch.randn(*shape, generator=gen, device=DEVICE) * scale
    return (normal(H, d, scale=2.0 / math.sqrt(d)), normal(H, scale=0.1), normal(C, H, scale=1.0 / math.sqrt(H)),
            normal(C, scale=0.1))


def _mlp(case, gen):
    weights = _network(case, gen)
    mlp = knng.Mlp(case["d"], case["hidden"], case["outputs"], seed=1, device=0)
    mlp.set_params(*[w.cpu().numpy() for w in weights])
    return mlp


def _edges(case, gen):
    """End points of a batch of graph edges: unit vectors, near pairs."""
    X = _points("sphere", case["edges"], case["d"], 256, "f32", gen)
    Y = X + 0.03 * torch.randn(X.shape, generator=gen, device=DEVICE)
    return torch.cat([X, Y / Y.norm(dim=1, keepdim=True)]).contiguous()


def _set_sizes(case):
    """Sizes of a batch's sets, spread over the logarithm of the range."""
    c = case["sets"]
    ratio = math.log(case["n_hi"] / case["n_lo"])
    out = []
    for i in range(c):
        u = ((i * 0.6180339887498949) % 1.0)
        out.append((int(case["n_lo"] * math.exp(ratio * u)), (64, 128, 256)[i % 3], 16 + (37 * i) % 241))
    return out


def prepare(case, seed):
    gen = _generator(seed)
    op = case["op"]
    state = dict(case=case)
    if op == "mlp_grad":
        state.update(mlp=_mlp(case, gen), pairs=_edges(case, gen))
        return state
    state["h"] = knng.Handle(0)
    if op == "batched":
        state["Xs"] = [_points("mixture", n, d, c, "f32", gen) for n, d, c in _set_sizes(case)]
        # one array holds all the sets' lists, back to back
        sizes, k = [X.shape[0] for X in state["Xs"]], case["k"]
        state["ids"] = torch.empty(sum(sizes), k, dtype=torch.int32, device=DEVICE)
        state["dists"] = torch.empty(sum(sizes), k, dtype=torch.float32, device=DEVICE)
        state["outs"] = list(zip(state["ids"].split(sizes), state["dists"].split(sizes)))
        return state
    X = _points(case["data"], case["n"], case["d"], case["centers"], case["dtype"], gen)
    state["X"] = X
    if op == "learned":
        state["mlp"] = _mlp(case, gen)
    elif op == "leaf":
        # the program's own divisions, next to the library's on the handle
        knng.knng_partition(X, case["T"], case["g"], TREE_SEED, h=state["h"])
        state["perm"] = _divisions(X, case["T"], case["g"], gen)
    elif op == "propagate":
        state["ids"], state["dists"] = _given_graph(X, case, gen)
    elif op == "exact_knn":
        state["queries"] = _sample(case, gen)
    return state


def _sample(case, gen):
    q = torch.randperm(case["n"], generator=gen, device=DEVICE)[:case["queries"]]
    return torch.sort(q).values.to(torch.int32).contiguous()


def run(state):
    c = state["case"]
    op = c["op"]
    if op == "build":
        return knng.knng_build(state["X"], c["k"], c["T"], c["g"], c["R"], TREE_SEED,
                               precision=PRECISION[c["precision"]], metric=METRIC[c["metric"]],
                               partitioner=PARTITIONER[c["partitioner"]], h=state["h"])
    if op == "batched":
        knng.knng_build_batched(state["Xs"], c["k"], c["T"], c["g"], c["R"], TREE_SEED,
                                precision=PRECISION[c["precision"]], outs=state["outs"], h=state["h"])
        return state["ids"], state["dists"]
    if op == "learned":
        return knng.knng_build_learned(state["mlp"], state["X"], c["k"], c["T"], c["g"], c["R"], TREE_SEED,
                                       precision=PRECISION[c["precision"]],
                                       partitioner=PARTITIONER[c["partitioner"]], h=state["h"])
    if op == "leaf":
        return knng.knng_leaf_knn(state["X"], c["T"], c["g"], state["perm"], c["k"],
                                  precision=PRECISION[c["precision"]], h=state["h"])
    if op == "propagate":
        if c["scheme"] == "best_first":
            return knng.knng_propagate_best_first(state["X"], state["ids"], c["budget"], rounds=c["R"], h=state["h"])
        return knng.knng_propagate(state["X"], state["ids"], state["dists"], rounds=c["R"], h=state["h"])
    if op == "exact_knn":
        return knng.knng_exact_knn(state["X"], state["queries"], c["k"], h=state["h"])
    if op == "mlp_grad":
        return state["mlp"].loss_grad(state["pairs"])
    raise ValueError(op)


# ------------------------------------------------------------------- work --
def _build_work(n, d, elem, k, T, g, levels_sizes):
    """Bytes: the rows in, the lists out.  Operations: one projection of
    every point per split level and tree, and one product per entry and pair
    of points that share a leaf."""
    depth = max(1, math.ceil(math.log2(max(1.0, n / g))))
    m = n / max(1, len(levels_sizes))
    return n * d * elem + 8 * n * k, T * n * depth * 2 * d + T * n * m * d


def work(case):
    op = case["op"]
    if op == "mlp_grad":
        N, d, H, C = 2 * case["edges"], case["d"], case["hidden"], case["outputs"]
        params = H * d + H + C * H + C
        # forward, weight gradients and the hidden gradient
        return {"bytes": 4 * (N * d + 2 * params), "flops": N * (4 * d * H + 6 * H * C)}
    if op == "batched":
        b = f = 0
        for n, d, _ in _set_sizes(case):
            nb, nf = _build_work(n, d, 4, case["k"], case["T"], case["g"], _leaf_sizes(n, case["g"]))
            b, f = b + nb, f + nf
        return {"bytes": b, "flops": f}
    n, d, k, elem = case["n"], case["d"], case["k"], ELEMENT_BYTES[case["dtype"]]
    if op in ("build", "learned"):
        b, f = _build_work(n, d, elem, k, case["T"], case["g"], _leaf_sizes(n, case["g"]))
        if op == "learned":
            f += 2 * n * case["hidden"] * (d + case["outputs"])
        return {"bytes": b, "flops": f}
    if op == "leaf":
        T = case["T"]
        m = n / len(_leaf_sizes(n, case["g"]))
        return {"bytes": n * d * elem + 4 * T * n + 8 * T * n * k, "flops": T * n * m * d}
    if op == "exact_knn":
        return {"bytes": n * d * elem + 4 * case["queries"] + 8 * case["queries"] * k,
                "flops": 2 * case["queries"] * n * d}
    # propagation: at least the k own neighbours' lists; one difference and
    # one product per entry of each point it has to score
    scored = case["budget"] if case["scheme"] == "best_first" else k * k // 4
    return {"bytes": n * d * elem + 16 * n * k, "flops": 3 * case["R"] * n * scored * d}


# ---------------------------------------------------------- 64-bit values --
def _propagated(X, ids, dist, k, rounds):
    """Synchronous first-order rounds in 64 bits (listed pairs keep their
    distances, others are computed)."""
    n, d = X.shape
    ids, dist = ids.long(), dist.double()
    step = max(1, (1 << 27) // ((k * k + k) * d))
    for _ in range(rounds):
        ni, nd = torch.empty_like(ids), torch.empty_like(dist)
        for s in range(0, n, step):
            own = torch.arange(s, min(n, s + step), device=DEVICE)
            far = ids[ids[own]].reshape(len(own), -1)
            diff = X[far].double() - X[own].double()[:, None, :]
            fd = (diff * diff).sum(2)
            # an id listed already keeps its distance: it sorts before
            # the computed copy and the later copy is dropped
            ni[own], nd[own] = _best(torch.cat([ids[own], far], 1), torch.cat([dist[own], fd], 1), own, k)
        ids, dist = ni, nd
    return dist


def _nearest(X, queries, k):
    q = queries.long()
    out = torch.empty(len(q), k, dtype=torch.float64, device=DEVICE)
    step = max(1, (1 << 28) // X.shape[0])
    for s in range(0, len(q), step):
        a = X[q[s:s + step]].double()
        parts = []
        for c in range(0, X.shape[0], 1 << 18):
            b = X[c:c + (1 << 18)].double()
            D = ((a * a).sum(1)[:, None] + (b * b).sum(1)[None, :] - 2.0 * (a @ b.T)).clamp_(min=0.0)
            hit = (q[s:s + step] >= c) & (q[s:s + step] < c + b.shape[0])
            rows = torch.nonzero(hit).ravel()
            D[rows, q[s:s + step][rows] - c] = math.inf
            parts.append(torch.topk(D, min(k, D.shape[1]), dim=1, largest=False).values)
        out[s:s + step] = torch.sort(torch.cat(parts, 1), dim=1).values[:, :k]
    return out


def _loss_and_gradient(weights, pairs):
    """The training loss (pull of neighbours relative to each output's
    variance, decorrelation, spread) and its gradient."""
    W = [w.double().requires_grad_(True) for w in weights]
    X = pairs.double()
    B = X.shape[0] // 2
    z = torch.tanh(torch.nn.functional.gelu(X @ W[0].T + W[1]) @ W[2].T + W[3])
    c = z - z.mean(0)
    var = (c * c).mean(0)
    pull = ((z[:B] - z[B:]) ** 2).mean(0)
    s = c / torch.sqrt(var + 1e-4)
    corr = s.T @ s / X.shape[0]
    off = corr - torch.diag(torch.diagonal(corr))
    loss = (pull / (var + 1e-4)).sum() + 0.05 * (off ** 2).sum() + ((1.0 - var) ** 2).sum()
    grads = torch.autograd.grad(loss, W)
    return float(loss.detach()), torch.cat([g.reshape(-1) for g in grads])


def exact(case, seed):
    # a build's divisions are decided by rounded projections, and a
    # best-first round by the order of rounded distances: their lists have
    # no value in 64 bits
    op = case["op"]
    gen = _generator(seed)
    if op == "mlp_grad":
        return _loss_and_gradient(_network(case, gen), _edges(case, gen))
    if op in ("build", "batched", "learned") or case.get("scheme") == "best_first":
        return None
    X = _points(case["data"], case["n"], case["d"], case["centers"], case["dtype"], gen)
    if op == "leaf":
        return None, _leaf_lists(X, _divisions(X, case["T"], case["g"], gen), case["g"], case["k"])[1]
    if op == "propagate":
        ids, dist = _given_graph(X, case, gen)
        return None, _propagated(X, ids, dist, case["k"], case["R"])
    if op == "exact_knn":
        return None, _nearest(X, _sample(case, gen), case["k"])
    return None

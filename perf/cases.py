"""Performance cases of the SLK library: what its users have it do, as plain
dicts, with the inputs, the call and the work of each.

A case's "op" is one of
  solve      slk.solve: kNN graph, sigma and Algorithm 1 on device data (with
             "sym" on the symmetric affinity)
  knn        slk.knn_graph on its own
  outer      one outer iteration of Algorithm 1 on a given graph, call by call:
             unary, bound_iterate, mode_update, energy
  meanshift  slk.mean_shift: the SLK-MS mode update with the assignments fixed
  modes0     slk.initial_modes: starting modes from the seeds' clusters
  seeds      slk.kmeanspp: K-means++ seeds
  batch      slk.solve_batched over many uneven problems
  serve      slk.Server: a burst of requests until all are done
Inputs are drawn on the GPU from the seed: the generators follow the shapes of
paper_1810_13044_gb300/inputs.py (blobs, an MNIST-shaped latent map, curved
manifolds with Zipf sizes, a mixture with one dominant cluster).
"""
import math
import random

import numpy as np
import torch

from paper_1810_13044_gb300 import slk


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 13)


def _randn(g, *shape, dtype=torch.float32):
    return torch.randn(*shape, generator=g, device="cuda", dtype=dtype)


def _labels(N, sizes, g):
    """Cluster ids in random order, `sizes` points each (summing to N)."""
    y = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"),
                                torch.tensor(sizes, device="cuda"))
    return y[torch.randperm(N, generator=g, device="cuda")]


def _sizes(N, weights):
    w = np.asarray(weights, dtype=np.float64)
    s = np.maximum((w / w.sum() * N).astype(np.int64), 1)
    s[int(np.argmax(s))] += N - int(s.sum())
    return s.tolist()


def _points(data, N, D, C, g):
    """(X float32 N x D, cluster ids) of a generator with C clusters."""
    if data == "blobs":
        y = _labels(N, _sizes(N, np.ones(C)), g)
        return 5.0 * _randn(g, C, D)[y] + _randn(g, N, D), y
    if data == "mixture":      # one cluster holds 70 % of the points
        w = np.concatenate([[0.7], np.full(max(C - 1, 1), 0.3 / max(C - 1, 1))])[:C]
        y = _labels(N, _sizes(N, w), g)
        return 4.0 * _randn(g, C, D)[y] + _randn(g, N, D), y
    if data == "mnist_like":   # 10 latent dimensions, two layers, features scaled to [0, 1]
        y = _labels(N, _sizes(N, np.ones(C)), g)
        mu = 3.0 * _randn(g, C, 10)
        W1, b1 = _randn(g, 256, 10) / math.sqrt(10.0), _randn(g, 256)
        W2, b2 = _randn(g, D, 256) / 16.0, 0.1 * _randn(g, D)
        X = torch.relu((mu[y] + _randn(g, N, 10)) @ W1.T + b1) @ W2.T + b2
        lo, hi = X.amin(0), X.amax(0)
        return ((X - lo) / torch.clamp(hi - lo, min=1e-6)).contiguous(), y
    # manifolds: curved, up to 8 dimensions, Zipf(1.1) sizes
    d = min(8, D)
    y = _labels(N, _sizes(N, np.arange(1, C + 1, dtype=np.float64) ** -1.1), g)
    c = 3.0 * _randn(g, C, D)
    U = torch.linalg.qr(_randn(g, C, D, d))[0]
    V = torch.linalg.qr(_randn(g, C, D, d))[0]
    X = torch.empty(N, D, device="cuda")
    for l in range(C):
        idx = torch.nonzero(y == l).flatten()
        t = _randn(g, idx.numel(), d)
        X[idx] = c[l] + t @ U[l].T + 0.3 * (t * t) @ V[l].T
    return X, y


def _one_per_cluster(y, C):
    """The first point of every cluster (int32 starting modes)."""
    N = y.numel()
    first = torch.full((C,), N, dtype=torch.int64, device="cuda")
    first.scatter_reduce_(0, y, torch.arange(N, device="cuda"), "amin")
    return first.to(torch.int32)


def _graph(y, C, k, heat, g):
    """A directed graph with k distinct neighbours of the own cluster per row
    (the shape of a kNN graph of clustered points in a random order)."""
    N = y.numel()
    order = torch.argsort(y, stable=True)
    size = torch.bincount(y, minlength=C)
    start = torch.cumsum(size, 0) - size
    pos = torch.empty_like(order)
    pos[order] = torch.arange(N, device="cuda")
    pos -= start[y]
    n = size[y]
    r = (torch.rand(N, generator=g, device="cuda", dtype=torch.float64) * (n - 1)).long()
    col = torch.empty(N, k, dtype=torch.int32, device="cuda")
    for j in range(k):
        # small clusters wrap into the next points of the order
        q = torch.where(n > k, start[y] + (pos + 1 + (r + j) % torch.clamp(n - 1, min=1)) % n,
                        (start[y] + pos + 1 + j) % N)
        col[:, j] = order[q].to(torch.int32)
    w = None
    if heat:
        w = 0.05 + 0.95 * torch.rand(N * k, generator=g, device="cuda")
    return torch.arange(N + 1, device="cuda") * k, col.reshape(-1).contiguous(), w


def _sigma(X, col, k):
    """Median distance over the edges of every 16th point or so."""
    N = X.shape[0]
    p = torch.arange(0, N, max(1, N // 20000), device="cuda")
    q = col.view(N, k)[p, 0].long()
    return float((X[p] - X[q]).square().sum(1).sqrt().median())


# ------------------------------------------------------------------ cases

def listed():
    return [
        # the smallest whole call: a small data set in the default precision, latency-bound
        dict(name="solve_2000x16_L5", op="solve", data="blobs", N=2000, D=16, L=5, k=5, heat=False,
             precision="fp32"),
        # the MNIST-shaped set of the benchmark (Table 1 of the paper)
        dict(name="solve_70000x784_L10", op="solve", data="mnist_like", N=70000, D=784, L=10, k=5,
             heat=False, precision="bf16_rerank"),
        # the benchmark's large set: many clusters of uneven sizes, heat affinity
        dict(name="solve_1000000x128_L100", op="solve", data="manifolds", N=1_000_000, D=128, L=100,
             k=10, heat=True, precision="bf16_rerank"),
        # a graph alone with the call's defaults (float32 tiles), ragged sizes, one dominant cluster
        dict(name="knn_30011x200_k12_fp32", op="knn", data="mixture", N=30011, D=200, C=12, k=12,
             heat=False, precision="fp32"),
        # one outer iteration step by step on a large graph in the given row order
        dict(name="outer_1000000x128_L100", op="outer", data="manifolds", N=1_000_000, D=128, L=100,
             k=10, heat=True, updates=6),
        # the same at a medium size with odd N and L, more updates
        dict(name="outer_150001x64_L37", op="outer", data="blobs", N=150001, D=64, L=37, k=7,
             heat=False, updates=40),
        # SLK-MS: mean-shift iterations of the MNIST-shaped set
        dict(name="meanshift_70000x784_L10", op="meanshift", data="mnist_like", N=70000, D=784, L=10,
             k=5, heat=False, iters=8),
        # starting modes (Section 4.2) of the MNIST-shaped set
        dict(name="modes0_70000x784_L10", op="modes0", data="mnist_like", N=70000, D=784, L=10),
        # K-means++ seeds of the large set
        dict(name="seeds_1000000x128_L100", op="seeds", data="manifolds", N=1_000_000, D=128, L=100),
        # the symmetric affinity of Prop. 1 (rows of uneven degree), odd sizes
        dict(name="solve_60001x50_L30_sym", op="solve", data="blobs", N=60001, D=50, L=30, k=8, heat=True,
             precision="bf16_rerank", sym=1),
        # many small uneven problems in one pass (the batched workload's ranges)
        dict(name="batch_64", op="batch", data="blobs", count=64, Nmin=500, Nmax=20000, Lmax=50, k=5,
             shapes=1),
        # a burst of requests to the server (the serving workload's ranges, bounded)
        dict(name="serve_16", op="serve", data="mnist_like", count=16, Nmin=1000, Nmax=50000, Lmax=100,
             k=6, shapes=2),
    ]


def _log_int(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    op = rng.choice(["solve", "solve", "solve", "knn", "outer", "outer", "meanshift", "modes0",
                     "seeds", "batch", "serve"])
    data = rng.choice(["blobs", "mnist_like", "manifolds"])
    if op == "solve":
        N, D = _log_int(rng, 1000, 400_000), _log_int(rng, 8, 800)
        while N * N * D > 2e13:
            N = int(N * 0.8)
        return dict(op=op, data=data, N=N, D=D, L=rng.randint(3, min(100, N // 40)),
                    k=rng.randint(3, 10), heat=rng.random() < 0.5,
                    precision="bf16_rerank" if N > 8000 else rng.choice(["fp32", "bf16_rerank"]),
                    sym=int(rng.random() < 0.2))
    if op == "knn":
        N, D = _log_int(rng, 2000, 60_000), _log_int(rng, 8, 800)
        while N * N * D > 1e12:
            N = int(N * 0.8)
        return dict(op=op, data=rng.choice([data, "mixture"]), N=N, D=D, C=rng.randint(2, 40),
                    k=rng.randint(1, 24), heat=rng.random() < 0.5, precision="fp32")
    if op == "outer":
        N, D, L = _log_int(rng, 10_000, 1_000_000), _log_int(rng, 8, 800), rng.randint(3, 128)
        while N * max(D, L) > 1.3e8:
            N = int(N * 0.8)
        return dict(op=op, data=data, N=N, D=D, L=L, k=rng.randint(3, 10), heat=rng.random() < 0.5,
                    updates=rng.randint(4, 40))
    if op == "meanshift":
        N, D, L = _log_int(rng, 5000, 200_000), _log_int(rng, 16, 1000), rng.randint(3, 40)
        while N * D * L > 8e8:
            N = int(N * 0.8)
        return dict(op=op, data=data, N=N, D=D, L=L, k=5, heat=False, iters=rng.randint(3, 12))
    if op == "modes0":
        N, D = _log_int(rng, 4000, 70_000), _log_int(rng, 16, 784)
        return dict(op=op, data=data, N=N, D=D, L=rng.randint(3, 40))
    if op == "seeds":
        N, D = _log_int(rng, 10_000, 1_000_000), _log_int(rng, 8, 784)
        while N * D > 1.3e8:
            N = int(N * 0.8)
        return dict(op=op, data=data, N=N, D=D, L=rng.randint(5, 100))
    if op == "batch":
        return dict(op=op, data="blobs", count=rng.randint(16, 64), Nmin=500, Nmax=20000,
                    Lmax=rng.randint(10, 50), k=rng.randint(4, 8), shapes=rng.randint(10, 10 ** 6))
    return dict(op=op, data="mnist_like", count=rng.randint(6, 20), Nmin=1000, Nmax=50000,
                Lmax=rng.randint(20, 100), k=rng.randint(5, 10), shapes=rng.randint(10, 10 ** 6))


def _problems(case):
    """(N, D, L) of each problem of a batch or burst: by the case alone."""
    r = random.Random(case["shapes"])
    dims = (9, 64, 256) if case["op"] == "batch" else (64, 512)
    out = []
    for _ in range(case["count"]):
        N = (r.randint(case["Nmin"], case["Nmax"]) if case["op"] == "batch"
             else _log_int(r, case["Nmin"], case["Nmax"]))
        out.append((N, r.choice(dims), r.randint(5, min(case["Lmax"], N // 50))))
    return out


def _params(case):
    return slk.default_params(affinity="heat" if case.get("heat") else "binary",
                              knn_precision=case.get("precision", "bf16_rerank"),
                              symmetrize=case.get("sym", 0))


def prepare(case, seed):
    g, op = _gen(seed), case["op"]
    s = dict(case=case)
    if op in ("batch", "serve"):
        shapes = _problems(case)
        s["Z"] = torch.empty(sum(N * L for N, _, L in shapes), device="cuda")
        s["labels"] = torch.empty(sum(N for N, _, _ in shapes), dtype=torch.int32, device="cuda")
        s["modes"] = torch.empty(sum(L for _, _, L in shapes), dtype=torch.int32, device="cuda")
        s["problems"], s["outs"], z, n, m = [], [], 0, 0, 0
        for N, D, L in shapes:
            X, y = _points(case["data"], N, D, L, g)
            s["problems"].append(dict(X=X, L=L, k=case["k"], lam=1.0, init_modes=_one_per_cluster(y, L)))
            s["outs"].append((s["Z"][z:z + N * L].view(N, L), s["labels"][n:n + N], s["modes"][m:m + L]))
            z, n, m = z + N * L, n + N, m + L
        s["params"] = slk.default_params(knn_precision="bf16_rerank")
        if op == "serve":
            s["server"] = slk.Server(max_slots=64, quantum=10, memory_bytes=4 << 30, params=s["params"])
        return s
    N, D = case["N"], case["D"]
    C = case["L"] if "L" in case else case["C"]
    X, y = _points(case["data"], N, D, C, g)
    s["X"] = X
    if op == "knn":
        s["sigma"] = 0.5 * float((X[:1000] - X[1000:2000]).square().sum(1).sqrt().median())
        return s
    if op == "seeds":
        r = np.random.default_rng(seed)
        s["first"], s["u"] = int(r.integers(N)), r.random(case["L"] - 1)
        return s
    s["modes"] = _one_per_cluster(y, C)
    if op == "solve":
        s["params"] = _params(case)
        return s
    if op == "modes0":
        # the width of a kNN graph's edges: within-cluster distances scaled down
        s["row_ptr"], col, _ = _graph(y, C, 1, False, g)
        s["sigma"] = 0.4 * _sigma(X, col, 1)
        return s
    k = case["k"]
    s["row_ptr"], s["col"], s["w"] = _graph(y, C, k, case["heat"], g)
    s["sigma"] = _sigma(X, s["col"], k)
    if op == "outer":
        L = case["L"]
        s["Z"], s["Zp"] = torch.empty(N, L, device="cuda"), torch.empty(N, L, device="cuda")
        return s
    M = X[s["modes"].long()]
    A = torch.empty(N, C, device="cuda")
    for a in range(0, N, 1 << 16):
        A[a:a + (1 << 16)] = torch.exp(-torch.cdist(X[a:a + (1 << 16)], M).square() / (2 * s["sigma"] ** 2))
    s["A"], s["M0"], s["Zp"] = A, M.clone(), torch.softmax(A, 1)
    return s


def run(s):
    case, op = s["case"], s["case"]["op"]
    if op == "solve":
        Z, labels, modes, st = slk.solve(s["X"], case["L"], case["k"], 1.0, s["modes"], params=s["params"])
        return dict(Z=Z, labels=labels, modes=modes, sigma=st["sigma"], energy=st["energy"],
                    outer=st["outer_iters"], inner=st["inner_iters_total"])
    if op == "knn":
        gr = slk.knn_graph(s["X"], case["k"], affinity="heat" if case["heat"] else "binary",
                           precision=case["precision"], sigma=s["sigma"])
        return dict(row_ptr=gr.row_ptr, col=gr.col_idx, dist2=gr.dist2, w=gr.w)
    if op == "outer":
        A, Z0 = slk.unary(s["X"], s["modes"], s["sigma"])
        Z, Zp = Z0, s["Zp"]
        slk.bound_iterate(A, s["row_ptr"], s["col"], s["w"], 1.0, Z, Zp, case["updates"])
        modes = s["modes"].clone()
        _, labels, key = slk.mode_update(A, Zp, s["row_ptr"], s["col"], s["w"], 1.0, modes)
        E = slk.energy(s["X"], labels, s["row_ptr"], s["col"], s["w"], case["L"], modes, s["sigma"], 1.0)
        return dict(A=A, Z=Z, Z_prev=Zp, labels=labels, modes=modes, key=key, energy=E)
    if op == "meanshift":
        M = s["M0"].clone()
        it, _, labels = slk.mean_shift(s["X"], s["A"], s["Zp"], s["row_ptr"], s["col"], s["w"], 1.0,
                                       s["sigma"], M, case["iters"])
        return dict(M=M, iters=it, labels=labels)
    if op == "modes0":
        modes, assign, dens = slk.initial_modes(s["X"], s["modes"], s["sigma"])
        return dict(modes=modes, assign=assign, density=np.array(dens))
    if op == "seeds":
        return dict(seeds=slk.kmeanspp(s["X"], case["L"], s["first"], s["u"]))
    if op == "batch":
        res = slk.solve_batched(s["problems"], params=s["params"], outs=s["outs"])
    else:
        tickets = [s["server"].submit(p, out=o) for p, o in zip(s["problems"], s["outs"])]
        done = s["server"].run_until_done(tickets)
        res = [done[t] for t in tickets]
    return dict(Z=s["Z"], labels=s["labels"], modes=s["modes"],
                energy=np.array([r[3]["energy"] for r in res]),
                inner=np.array([r[3]["inner_iters_total"] for r in res]))


def _solve_work(N, D, L, k, updates, outers):
    """A solve: the distances of all pairs, then the iterations; X and the
    outputs once, the iterate once per update."""
    e = 4 * N * (D + 2 * L + 2 * k + 2)
    return dict(flops=2.0 * N * N * D + outers * 5.0 * N * D * L + updates * N * L * (2 * k + 6),
                bytes=float(e + outers * 4 * N * D + updates * 4 * N * (3 * L + k)))


def work(case):
    op = case["op"]
    if op in ("batch", "serve"):
        ws = [_solve_work(N, D, L, case["k"], 10, 1) for N, D, L in _problems(case)]
        return dict(bytes=sum(w["bytes"] for w in ws), flops=sum(w["flops"] for w in ws))
    N, D, k, L = case["N"], case["D"], case.get("k", 0), case.get("L", 0)
    if op == "solve":
        return _solve_work(N, D, L, k, 6, 1)
    if op == "knn":
        return dict(flops=2.0 * N * N * D, bytes=float(4 * N * (D + 2 * k + 2)))
    if op == "outer":
        u = case["updates"]
        return dict(flops=3.0 * N * D * L + u * N * L * (2 * k + 6) + N * L * (2 * k + 6),
                    bytes=float(4 * N * (2 * D + 2 * L) + (u + 1) * 4 * N * (3 * L + k + 2)))
    if op == "meanshift":
        # 5 operations per point, label and feature; X once per iteration
        it = case["iters"]
        return dict(flops=5.0 * N * D * L * it, bytes=float(it * 4 * N * D + 4 * N * 3 * L))
    if op == "modes0":
        return dict(flops=2.0 * N * N * D + 3.0 * N * D * L, bytes=float(4 * N * (D + 1)))
    # seeds: X once, every new seed against the smallest distance so far
    return dict(flops=3.0 * N * D * (L - 1), bytes=float(4 * N * D + 16 * N))


# ------------------------------------------------------------------ 64 bits

def _unary64(X, modes, sigma):
    A = torch.empty(X.shape[0], modes.numel(), device="cuda", dtype=torch.float64)
    Xd = X.double()
    for l, m in enumerate(modes.tolist()):
        A[:, l] = torch.exp(-(Xd - Xd[m]).square().sum(1) / (2 * sigma * sigma))
    return A


def _pairwise64(Z, col, w, k):
    b = torch.zeros_like(Z)
    c = col.view(-1, k).long()
    for j in range(k):
        b += Z[c[:, j]] if w is None else Z[c[:, j]] * w.view(-1, k)[:, j:j + 1].double()
    return b


def exact(case, seed):
    op = case["op"]
    if op in ("solve", "batch", "serve", "seeds"):
        return None   # seeds are whole numbers; a whole solve's path follows its rounding
    N = case["N"]
    if op == "modes0" and N * N * case["D"] > 4.2e12:
        return None
    s = prepare(case, seed)
    k = case.get("k", 0)
    sigma = float(np.float32(s["sigma"])) if "sigma" in s else 0.0
    if op == "knn":
        X = s["X"].double()
        X -= X.mean(0)
        n2 = X.square().sum(1)
        d2 = torch.empty(N, k, device="cuda", dtype=torch.float64)
        for a in range(0, N, 2048):
            d = n2[a:a + 2048, None] + n2 - 2 * X[a:a + 2048] @ X.T
            d[torch.arange(d.shape[0]), torch.arange(a, a + d.shape[0])] = math.inf
            c = d.topk(k, largest=False).indices
            for j in range(k):
                d2[a:a + 2048, j] = (X[a:a + 2048] - X[c[:, j]]).square().sum(1)
        d2 = d2.sort(1).values.reshape(-1)
        w = torch.exp(-d2 / (2 * sigma * sigma)) if case["heat"] else None
        return dict(row_ptr=None, col=None, dist2=d2, w=w)
    if op == "modes0":
        X = s["X"].double()
        X -= X.mean(0)
        n2 = X.square().sum(1)
        seeds = s["modes"].long()
        a = (n2[:, None] + n2[seeds] - 2 * X @ X[seeds].T).argmin(1)
        dens = []
        for l in range(case["L"]):
            mem = torch.nonzero(a == l).flatten()
            f = torch.zeros(N, device="cuda", dtype=torch.float64)
            for b in range(0, mem.numel(), 2048):
                m = mem[b:b + 2048]
                d = (n2[m, None] + n2 - 2 * X[m] @ X.T).clamp_(min=0)
                f += d.mul_(-1 / (2 * sigma * sigma)).exp_().sum(0)
            dens.append(float(f.max()))
        return dict(modes=None, assign=None, density=np.array(dens))
    if op == "meanshift":
        S = s["A"].double() + _pairwise64(s["Zp"].double(), s["col"], s["w"], k)
        lz = torch.log_softmax(S, 1)
        X, M = s["X"].double(), s["M0"].double()
        for _ in range(case["iters"]):
            new = torch.empty_like(M)
            for l in range(M.shape[0]):
                t = lz[:, l] - (X - M[l]).square().sum(1) / (2 * sigma * sigma)
                t = torch.exp(t - t.max())
                new[l] = (t @ X) / t.sum()
            M = new
        return dict(M=M, iters=None, labels=None)
    # outer
    A = _unary64(s["X"], s["modes"], sigma)
    Z, Zp = torch.softmax(A, 1), None
    for _ in range(case["updates"]):
        Zp, Z = Z, torch.softmax(A + _pairwise64(Z, s["col"], s["w"], k), 1)
    lz = torch.log_softmax(A + _pairwise64(Zp, s["col"], s["w"], k), 1)
    key, modes = lz.max(0)
    labels = lz.argmax(1)
    X = s["X"].double()
    E = -torch.exp(-(X - X[modes[labels]]).square().sum(1) / (2 * sigma * sigma)).sum()
    cut = (labels[s["col"].long()].view(N, k) != labels[:, None]).double()
    if s["w"] is not None:
        cut *= s["w"].view(N, k).double()
    return dict(A=A, Z=Z, Z_prev=Zp, labels=None, modes=None, key=key, energy=float(E + cut.sum()))

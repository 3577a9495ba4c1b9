"""The tensor-core candidate sweep and the sort by regions in front of it.

Both precisions must give the same graph (a full float32 scan), and the
float32 tiles neither sort the points nor leave tiles out, so every form of
input goes through both: clustered data, one cluster (nothing can be left
out), points in sorted order, duplicates, far outliers, all points equal;
sizes at the edges of tiles, feature counts of every K loop (folded norms,
resident rows, plain), k at the edges of the lists.
"""
import numpy as np
import pytest

import oracle
from paper_1810_13044_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def slk():
    from paper_1810_13044_gb300 import build, slk as _slk
    build.build()
    return _slk


def points(kind, N, D, seed):
    g = inputs.rng(seed)
    if kind == "one":
        return g.normal(size=(N, D)).astype(np.float32)
    if kind == "equal":
        return np.full((N, D), 1.5, np.float32)
    X, y = inputs.blobs(N=N, D=D, n_blobs=23, centre_var=25.0, seed=seed)
    if kind == "sorted":
        X = np.ascontiguousarray(X[np.argsort(y, kind="stable")])
    if kind == "duplicates":
        X[N // 2:] = X[: N - N // 2]
    if kind == "outliers":
        X[:40] *= np.float32(50.0)
    return X


@pytest.mark.parametrize("kind", ["blobs", "one", "sorted", "duplicates", "outliers"])
@pytest.mark.parametrize("N,D,k", [(32768, 64, 5), (32641, 50, 10), (33025, 9, 1), (24000, 130, 24),
                                   (20225, 257, 7), (16500, 520, 6), (40001, 3, 12)])
def test_sorted_sweep_equals_float32_tiles(slk, kind, N, D, k):
    X = torch.from_numpy(points(kind, N, D, N + k)).cuda()
    a = slk.knn_graph(X, k, precision="bf16_rerank")
    b = slk.knn_graph(X, k, precision="fp32")
    assert torch.equal(a.dist2, b.dist2)
    assert torch.equal(a.col_idx, b.col_idx)
    assert torch.equal(a.row_ptr, b.row_ptr)


def test_all_points_equal(slk):
    """Every distance ties: each row's neighbours are the smallest indices."""
    N, k = 20000, 6
    X = torch.from_numpy(points("equal", N, 40, 0)).cuda()
    g = slk.knn_graph(X, k, precision="bf16_rerank")
    col = g.col_idx.cpu().numpy().reshape(N, k)
    want = np.arange(k)[None, :] + (np.arange(k)[None, :] >= np.arange(N)[:, None])
    np.testing.assert_array_equal(col, want)
    assert float(g.dist2.abs().max()) == 0.0


def test_two_term_stage_after_a_sorted_sweep(slk):
    """Rows the sorted sweep leaves open get their operand back in the points'
    order: two clusters far from the mean, sampled rows against the oracle."""
    N, D, k = 120000, 32, 8
    g = inputs.rng(5)
    X = g.normal(size=(N, D)).astype(np.float32)
    X[g.permutation(N)[: N // 2], 1] += np.float32(220.0)
    gr = slk.knn_graph(torch.from_numpy(X).cuda(), k, precision="bf16_rerank")
    assert gr.stage_rows[0] > 1000, gr.stage_rows
    rows = g.choice(N, size=300, replace=False)
    o_idx, o_d2 = oracle.knn(X, k, rows=rows)
    got = gr.col_idx.cpu().numpy().reshape(N, k)[rows]
    d2 = gr.dist2.cpu().numpy().reshape(N, k)[rows]
    np.testing.assert_allclose(d2, o_d2, rtol=2.0 * (D + 8) * 2.0 ** -24)
    assert (got != o_idx).any(1).sum() <= 6   # swaps of near-equal distances


def test_least_workspace_gives_the_same_solution(slk):
    """A server whose arena holds exactly the request's least need builds its
    graph from the small plan (short lists, whole row blocks, no sort)."""
    X, y = inputs.blobs(N=30000, D=48, n_blobs=12, centre_var=25.0, seed=3)
    init = torch.tensor([int(np.nonzero(y == c)[0][0]) for c in range(12)], dtype=torch.int32).cuda()
    Xd = torch.from_numpy(X).cuda()
    params = slk.default_params(knn_precision="bf16_rerank")
    pr = dict(X=Xd, L=12, k=6, lam=1.0, init_modes=init)
    big = slk.Server(memory_bytes=1 << 30, params=params)
    need = big.request_bytes(pr)
    want = big.run_until_done([big.submit(pr)])
    small = slk.Server(memory_bytes=need, params=params)
    got = small.run_until_done([small.submit(pr)])
    (Z0, l0, m0, s0), (Z1, l1, m1, s1) = want.popitem()[1], got.popitem()[1]
    assert torch.equal(Z0, Z1) and torch.equal(l0, l1) and torch.equal(m0, m1)
    assert s0["sigma"] == s1["sigma"]
    big.close()
    small.close()


def test_all_points_equal_sorted(slk):
    """The same above the work size from which the points are sorted: no border
    between any two pivots, and every row of the first sweep given up on ties."""
    N, D, k = 40000, 40, 6
    X = torch.from_numpy(points("equal", N, D, 0)).cuda()
    g = slk.knn_graph(X, k, precision="bf16_rerank")
    col = g.col_idx.cpu().numpy().reshape(N, k)
    want = np.arange(k)[None, :] + (np.arange(k)[None, :] >= np.arange(N)[:, None])
    np.testing.assert_array_equal(col, want)
    assert float(g.dist2.abs().max()) == 0.0


def test_refused_workspace_is_asked_for_again(slk):
    """A context that once could not have the larger workspace takes the least
    one, and the larger one once the memory is free again."""
    N, D, k = 200000, 64, 10
    MB = 1 << 20
    X = torch.from_numpy(points("blobs", N, D, 1)).cuda()

    def spare():                  # leaves room for the outputs in torch's cache
        outs = [torch.empty(4 * N * k, device="cuda") for _ in range(2)]
        del outs

    def grown(ctx):               # device memory a graph takes beyond its outputs
        free = torch.cuda.mem_get_info()[0]
        g = slk.knn_graph(X, k, precision="bf16_rerank", ctx=ctx)
        torch.cuda.synchronize()
        return free - torch.cuda.mem_get_info()[0], g

    a = slk.Context()
    grown(a)                      # (first launches load code)
    a.close()
    a, b = slk.Context(), slk.Context()
    spare()
    full, g0 = grown(a)
    a.close()
    torch.cuda.empty_cache()
    spare()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (full - 24 * MB), dtype=torch.uint8, device="cuda")
    try:
        less, g1 = grown(b)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert 0 < less < full - 24 * MB
    spare()
    more, g2 = grown(b)
    assert more > 24 * MB
    for g in (g1, g2):
        assert torch.equal(g.col_idx, g0.col_idx) and torch.equal(g.dist2, g0.dist2)
    b.close()

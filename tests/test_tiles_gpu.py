"""Edges of the float32 distance tiles (lists brought up to date by sorting or
by insertion) and of the unary kernel's passes and copies."""
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


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("order", ["away", "towards", "random", "equal"])
@pytest.mark.parametrize("N,D,k", [(127, 1, 1), (128, 15, 7), (129, 16, 8), (257, 17, 9), (1025, 3, 16),
                                   (3001, 33, 24)])
def test_float32_tiles_exact(slk, order, N, D, k):
    """Integer coordinates: every distance exact, so the graph is the oracle's
    entry by entry whichever way the columns arrive (nearest first, nearest
    last: every column enters every list, random, all equal)."""
    if order == "equal":
        X = np.ones((N, D))
    else:
        X = inputs.rng(N).integers(0, 4, size=(N, D)).astype(np.float64)
        X[:, 0] = np.arange(N) % 64
        if order == "random":
            X = X[inputs.rng(k).permutation(N)]
        else:
            X = X[np.argsort(X[:, 0], kind="stable")][:: 1 if order == "away" else -1]
    X = X.astype(np.float32)
    o_idx, o_d2 = oracle.knn(X, k)
    g = slk.knn_graph(dev(X), k, precision="fp32")
    np.testing.assert_array_equal(g.col_idx.cpu().numpy().reshape(N, k), o_idx)
    np.testing.assert_array_equal(g.dist2.cpu().numpy().reshape(N, k).astype(np.float64), o_d2)


@pytest.mark.parametrize("shift", [0, 1])   # X on a 16-byte boundary, or 4 bytes past one
@pytest.mark.parametrize("N,D,L", [(256, 4, 8), (257, 36, 9), (129, 32, 28), (130, 35, 32), (128, 64, 33),
                                   (300, 12, 57), (255, 2, 64), (301, 33, 256)])
def test_unary_passes_and_copies(slk, N, D, L, shift):
    g = inputs.rng(N + D + L)
    X = g.normal(size=(N, D)).astype(np.float32)
    modes = g.choice(N, size=L, replace=L > N).astype(np.int32)
    sig = float(np.sqrt(D))
    buf = torch.empty(N * D + shift, dtype=torch.float32, device="cuda")
    Xd = buf[shift:].view(N, D)
    Xd.copy_(torch.from_numpy(X))
    A, Z0 = slk.unary(Xd, dev(modes), sig)
    Ao = oracle.unary(X, modes, sig)
    assert np.abs(A.cpu().numpy() - Ao).max() <= 1e-6
    assert np.abs(Z0.cpu().numpy() - oracle.softmax_rows(Ao)).max() <= 1e-6


@pytest.mark.parametrize("N,D,L", [(127, 31, 1), (300, 32, 4), (128, 32, 5), (129, 33, 8), (1000, 9, 7), (255, 16, 9),
                                   (256, 32, 32), (300, 64, 28), (131, 8, 33), (131, 40, 40), (140, 7, 96),
                                   (257, 33, 255)])
def test_unary_rows_of_both_outputs(slk, N, D, L):
    """One step (a single buffer, the softmax in place), several of one pass (in the
    other buffer) and several passes (read back), with one to eight label groups;
    A alone is the same."""
    g = inputs.rng(N + D + L)
    X = g.normal(size=(N, D)).astype(np.float32)
    modes = g.choice(N, size=L, replace=False).astype(np.int32)
    sig = float(np.sqrt(D))
    A, Z0 = slk.unary(dev(X), dev(modes), sig)
    Ao = oracle.unary(X, modes, sig)
    assert np.abs(A.cpu().numpy() - Ao).max() <= 1e-6
    assert np.abs(Z0.cpu().numpy() - oracle.softmax_rows(Ao)).max() <= 1e-6
    assert torch.equal(A, slk.unary(dev(X), dev(modes), sig, with_z0=False)[0])


@pytest.mark.parametrize("N,D,k", [(81, 5, 24), (130, 100, 7), (1000, 128, 24), (3001, 200, 10), (2500, 300, 24),
                                   (2000, 900, 6), (1500, 1100, 24)])
@pytest.mark.parametrize("groups", [1, 3, 5])
@pytest.mark.parametrize("precision", ["bf16_rerank", "fp32"])
def test_few_rows_rescanned(slk, N, D, k, groups, precision):
    """Points with 79 copies: their neighbours tie at distance 0, so no list certifies
    them and they are rescanned exactly, fewer rows than CTAs, a row's columns over
    one range or many.  Integer coordinates: the oracle's graph entry by entry."""
    g = inputs.rng(N + D)
    X = g.integers(0, 4, size=(N, D)).astype(np.float32)
    groups = min(groups, N // 80)
    at = g.permutation(N)[: 80 * groups].reshape(groups, 80)
    for a in at:
        X[a] = X[a[0]]
    o_idx, o_d2 = oracle.knn(X, k)
    gr = slk.knn_graph(dev(X), k, precision=precision)
    assert gr.stage_rows[2] >= 80 * groups
    np.testing.assert_array_equal(gr.col_idx.cpu().numpy().reshape(N, k), o_idx)
    np.testing.assert_array_equal(gr.dist2.cpu().numpy().reshape(N, k).astype(np.float64), o_d2)

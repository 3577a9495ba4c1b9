"""Sparse affinities whose rows differ in degree: the z-updates over rows from
empty to hubs (their own windows above 48 entries; more hubs than a block
lists), and the symmetrisation of long in-lists (ranked by a block above 48)."""
import numpy as np
import pytest

import oracle
from paper_1810_13044_gb300 import inputs
from parity_checks import Z_TOL

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def slk():
    from paper_1810_13044_gb300 import build, slk as _slk
    build.build()
    return _slk


def dev(a):
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _graph(N, degrees, seed, weighted):
    """Row p has degrees[p % len(degrees)] random entries."""
    g = inputs.rng(seed)
    deg = np.resize(np.asarray(degrees, np.int64), N)
    rp = np.concatenate([[0], np.cumsum(deg)])
    ci = g.integers(0, N, size=int(rp[-1])).astype(np.int32)
    w = g.uniform(0.1, 1.0, size=int(rp[-1])).astype(np.float32) if weighted else None
    return rp, ci, w


EDGES = [0, 1, 2, 7, 8, 9, 15, 16, 17, 31, 33, 47, 48, 49, 63, 64, 65, 97, 300]


@pytest.mark.parametrize("N,degrees,L,weighted", [
    (2, [0, 1], 3, False),           # (no entry at all is refused: a NULL col_idx)
    (1, [60], 30, True),
    *[(1203, EDGES, L, bool(L % 2)) for L in (1, 2, 3, 5, 9, 16, 17, 30, 33, 64, 65, 128, 200, 256)],
    (30011, [0, 0, 0, 700] + [3] * 40, 30, True),
    (300007, [49], 2, False),        # every row a hub: more than a block lists
    (60013, [5] * 4000 + [900], 12, True),
])
def test_bound_iterate_rows_of_any_degree(slk, N, degrees, L, weighted):
    rp, ci, w = _graph(N, degrees, N + L, weighted)
    deg = np.diff(rp)
    A = inputs.random_unary(N, L, seed=L)
    Z0 = inputs.random_simplex_rows(N, L, seed=L + 1)
    lam = 1.3 / max(deg.mean(), 1.0)
    for iters in (1, 4):
        Z = dev(Z0)
        Zp = torch.empty_like(Z)
        it, _ = slk.bound_iterate(dev(A), dev(rp), dev(ci), dev(w), lam, Z, Zp, iters, tol=-1.0)
        Zo, Zpo, _, _ = oracle.bound_iterate(A, rp, ci, w, lam, Z0, iters)
        assert it == iters
        assert np.abs(Z.cpu().numpy() - Zo).max() <= Z_TOL
        assert np.abs(Zp.cpu().numpy() - Zpo).max() <= Z_TOL


@pytest.mark.parametrize("N,hubs,weighted", [(49, 1, True), (50, 1, True), (51, 2, False),
                                             (700, 3, True), (9000, 5, True)])
def test_symmetrize_long_in_lists(slk, N, hubs, weighted):
    """Every point lists the first `hubs` points and two at random, one of
    them twice: in-lists of about N entries with repeated sources."""
    g = inputs.rng(N)
    ci = np.concatenate([np.tile(np.arange(hubs), (N, 1)), g.integers(0, N, (N, 2))], 1)
    ci = np.concatenate([ci, ci[:, -1:]], 1)
    rp = np.arange(N + 1, dtype=np.int64) * ci.shape[1]
    ci = ci.reshape(-1).astype(np.int32)
    w = g.uniform(0.1, 1.0, size=ci.size).astype(np.float32) if weighted else None
    g_rp, g_ci, g_w = slk.symmetrize(dev(rp), dev(ci), dev(w), N)
    o_rp, o_ci, o_w = oracle.symmetrize(rp, ci, w, N)
    np.testing.assert_array_equal(g_rp.cpu().numpy(), o_rp)
    np.testing.assert_array_equal(g_ci.cpu().numpy(), o_ci)
    # sums of up to four float32 terms, then one rounding
    np.testing.assert_allclose(g_w.cpu().numpy(), o_w, rtol=2 ** -21, atol=0)

"""GPU parity of the starting modes (Section 4.2: nearest-seed assignment,
then the mode definition of Eq. (1)) through the C-ABI against the FP64
oracle.

Integer results are compared exactly except where float rounding decides
them between near-equal candidates:
  assignment: the oracle's float64 squared distances to the two seeds agree
    within 1e-6 relative (the GPU sums float32 squares of float32
    differences in chunks of 32, in float64);
  modes: the oracle's cluster density at the GPU's mode is within DENS_RTOL
    of the oracle's maximum.
DENS_RTOL: the reported densities (and the final choice among the
certified candidates) come from float32 differences whose squares are
summed in float32 chunks of 8 and then in float64: d2 is within ~9u
relative (u = 2^-24), so a kernel value k = exp(-d2 / (2 sigma^2)) within
9u d2 / (2 sigma^2) relative; the terms that carry weight have d2 below
~40 sigma^2, which bounds the relative error of a density by ~1.1e-5.
"""
import numpy as np
import pytest

import oracle
from paper_1810_13044_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DENS_RTOL = 2e-5


@pytest.fixture(scope="module")
def slk():
    from paper_1810_13044_gb300 import build, slk as _slk
    build.build()
    return _slk


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    return t.detach().cpu().numpy()


def _check_assign(X, seeds, g_assign, o_assign):
    diff = np.nonzero(g_assign != o_assign)[0]
    for p in diff:
        d = ((X[p].astype(np.float64) - X[seeds[[g_assign[p], o_assign[p]]]].astype(np.float64)) ** 2).sum(1)
        assert abs(d[0] - d[1]) <= 1e-6 * max(d.max(), 1e-30), (p, d)
    assert len(diff) <= max(1, len(g_assign) // 1000)


def _check_modes(X, sig, g_modes, g_dens, o_modes, o_dens, o_assign):
    L = len(o_modes)
    for l in range(L):
        if o_dens[l] == 0.0:                      # empty cluster: keeps its seed
            assert g_dens[l] == 0.0 and g_modes[l] == o_modes[l]
            continue
        if g_modes[l] != o_modes[l]:
            f = oracle.cluster_density(X, o_assign, l, sig, np.array([g_modes[l]]))[0]
            assert f >= o_dens[l] * (1 - DENS_RTOL), (l, g_modes[l], o_modes[l], f, o_dens[l])
        assert g_dens[l] == pytest.approx(o_dens[l], rel=DENS_RTOL)


@pytest.mark.parametrize("N,D,L,seed", [
    (2000, 16, 5, 1810),      # the 2000 x 16 blobs workload
    (3000, 784, 10, 2),       # the 70000 x 784 shape
    (300, 7, 3, 3),           # ragged tiles, D % 16 != 0
    (1500, 64, 40, 4),        # many clusters, uneven sizes
    (129, 130, 1, 5),         # one cluster
    (1, 3, 1, 6),             # one point
])
def test_initial_modes_match_oracle(slk, N, D, L, seed):
    if (N, D) == (2000, 16):
        X, _ = inputs.blobs(seed=seed)
    elif D == 784:
        X, _ = inputs.mnist_like(N=N, seed=seed)
    else:
        X, _ = inputs.blobs(N=N, D=D, n_blobs=max(L, 1), centre_var=9.0, seed=seed)
    seeds = inputs.kmeanspp(X, L, seed=seed) if N > 1 else np.zeros(1, np.int32)
    sig = float(0.4 * np.sqrt(2.0 * D))
    o_modes, o_assign, o_dens = oracle.initial_modes(X, seeds, sig)
    st = {}
    g_modes, g_assign, g_dens = slk.initial_modes(dev(X), dev(seeds), sig, stats=st)
    _check_assign(X, seeds, host(g_assign), o_assign)
    _check_modes(X, sig, host(g_modes), np.array(g_dens), o_modes, o_dens, o_assign)
    print(f"initial modes N={N} D={D} L={L}: {st['candidates']} exact recomputes")
    assert 1 <= st["candidates"] <= N * L


def test_initial_modes_duplicate_and_empty_cluster(slk):
    g = inputs.rng(9)
    X = g.normal(size=(400, 6)).astype(np.float32)
    X[250] = X[17]                                # a duplicate: wins under a narrow kernel
    seeds = np.array([17, 17, 300], np.int32)     # label 1 ties with label 0: empty
    o_modes, o_assign, o_dens = oracle.initial_modes(X, seeds, 1e-3)
    g_modes, g_assign, g_dens = slk.initial_modes(dev(X), dev(seeds), 1e-3)
    np.testing.assert_array_equal(host(g_assign), o_assign)
    np.testing.assert_array_equal(host(g_modes), o_modes)
    assert host(g_modes)[1] == 17 and g_dens[1] == 0.0
    assert g_dens[0] == pytest.approx(2.0, rel=1e-6)


def test_initial_modes_full_size_sampled(slk):
    """The 70000 x 784, L=10 workload: the oracle's assignment in full, then
    the oracle's cluster density at the GPU's mode and at sampled points of
    each cluster (its seed among them)."""
    X, _ = inputs.mnist_like()
    L = 10
    seeds = inputs.kmeanspp(X, L, seed=1810)
    sig = 3.0
    st = {}
    g_modes, g_assign, g_dens = slk.initial_modes(dev(X), dev(seeds), sig, stats=st)
    gm, ga = host(g_modes), host(g_assign)
    print(f"initial modes full size: {st['candidates']} exact recomputes")
    assert st["candidates"] < X.shape[0]        # the bound leaves a small candidate set
    o_assign = np.empty(X.shape[0], np.int32)
    d = np.full(X.shape[0], np.inf)
    X64 = X.astype(np.float64)
    for l, s in enumerate(seeds):
        dl = ((X64 - X64[s]) ** 2).sum(1)
        better = dl < d
        o_assign[better] = l
        d[better] = dl[better]
    _check_assign(X, seeds, ga, o_assign)
    rng = inputs.rng(10)
    for l in range(L):
        members = np.nonzero(o_assign == l)[0]
        sample = np.concatenate([[gm[l], seeds[l]], rng.choice(members, size=min(40, len(members)),
                                                               replace=False)])
        f = oracle.cluster_density(X, o_assign, l, sig, sample)
        assert f[0] >= f.max() * (1 - DENS_RTOL)
        assert g_dens[l] == pytest.approx(f[0], rel=DENS_RTOL)


def test_solve_with_refined_start_matches_oracle(slk):
    """slk_solve with refine_init: Algorithm 1 from the starting modes."""
    X, _ = inputs.blobs()
    L, k, lam = 5, 5, 1.0
    seeds = inputs.kmeanspp(X, L, seed=1810)
    idx, d2 = oracle.knn(X, k)
    sig = oracle.sigma(d2)
    o_start, _, _ = oracle.initial_modes(X, seeds, sig)
    ref = oracle.solve(X, L, k, lam, o_start, sig=sig)
    p = slk.default_params(refine_init=1)
    Z, labels, modes, st = slk.solve(dev(X), L, k, lam, dev(seeds), sigma=sig, params=p)
    np.testing.assert_array_equal(host(modes), ref["modes"])
    np.testing.assert_array_equal(host(labels), ref["labels"])
    assert np.abs(host(Z) - ref["Z"]).max() <= 1e-5
    assert st["energy"] == pytest.approx(ref["E"], rel=1e-6)


# ------------------------------------------------------------ K-means++ seeds

@pytest.mark.parametrize("case", ["blobs", "mixture", "mnist_like", "manifolds", "duplicates"])
def test_kmeanspp_matches_oracle(slk, case):
    """GPU K-means++ from the same draws gives the oracle's seeds index for
    index (and the numpy recipe's)."""
    if case == "blobs":
        X, _ = inputs.blobs()
        L, seed = 5, 1810
    elif case == "mixture":
        X, _ = inputs.mixture(20000, 9, 50, seed=8)
        L, seed = 50, 8
    elif case == "mnist_like":
        X, _ = inputs.mnist_like(N=6000)
        L, seed = 10, 1810
    elif case == "manifolds":
        X, _ = inputs.manifolds(N=20000)
        L, seed = 100, 1810
    else:   # every point repeated: exact zero distances, and an all-zero draw
        base = inputs.rng(3).normal(size=(7, 5)).astype(np.float32)
        X = np.repeat(base, 40, axis=0)
        L, seed = 12, 3
    first, u = inputs.kmeanspp_draws(X.shape[0], L, seed)
    want = oracle.kmeanspp(X, L, first, u)
    got = slk.kmeanspp(torch.from_numpy(X).cuda(), L, first, u).cpu().numpy()
    np.testing.assert_array_equal(got, want)
    np.testing.assert_array_equal(got, inputs.kmeanspp(X, L, seed=seed))


def test_kmeanspp_rejects_bad_draws(slk):
    X = torch.zeros(10, 3, device="cuda")
    with pytest.raises(slk.SlkError, match="INVALID_ARG"):
        slk.kmeanspp(X, 3, 0, [0.5, 1.0])
    with pytest.raises(slk.SlkError, match="INVALID_ARG"):
        slk.kmeanspp(X, 3, 10, [0.5, 0.5])
    with pytest.raises(slk.SlkError, match="INVALID_ARG"):
        slk.kmeanspp(X, 11, 0, [0.5] * 10)


@pytest.mark.parametrize("N,D,L", [(255, 1, 9), (256, 3, 40), (257, 4, 40), (1000, 8, 60), (5000, 17, 300),
                                   (3001, 36, 50), (3001, 64, 50), (2000, 132, 25), (400001, 12, 20)])
@pytest.mark.parametrize("shift,scale", [(0.0, 1.0), (3e4, 1.0), (0.0, 1e-22), (0.0, 3e18)])
def test_kmeanspp_screened_distances(slk, N, D, L, shift, scale):
    """The bounds that skip float64 distances change no seed: lanes per point
    4 to 32, tile edges, data far from the origin (the float32 distances are
    coarse), and scales at which float32 squares underflow or overflow (the
    bounds must step aside).  Index for index against the oracle."""
    X, _ = inputs.blobs(N=N, D=D, n_blobs=8, centre_var=25.0, seed=N + D)
    X = ((X + np.float32(shift)) * np.float32(scale)).astype(np.float32)
    first, u = inputs.kmeanspp_draws(N, L, seed=D)
    got = host(slk.kmeanspp(dev(X), L, first, u))
    np.testing.assert_array_equal(got, oracle.kmeanspp(X, L, first, u))


@pytest.mark.parametrize("N,D,L,sigma", [(3000, 5, 12, 0.3), (3000, 5, 12, 3.0), (3000, 5, 12, 40.0),
                                         (2049, 33, 40, 2.0), (4000, 2, 3, 0.05), (1500, 7, 1, 1.0)])
def test_initial_modes_other_clusters_left_out(slk, N, D, L, sigma):
    """Row blocks of other clusters are left out only where they cannot hold
    the maximiser: overlapping clusters and widths from far below to far above
    the clusters' distances, against the oracle over all pairs."""
    X, _ = inputs.blobs(N=N, D=D, n_blobs=max(2, L // 2), centre_var=4.0, seed=N + L)
    seeds = inputs.kmeanspp(X, L, seed=L)
    o_modes, o_assign, o_dens = oracle.initial_modes(X, seeds, sigma)
    g_modes, g_assign, g_dens = slk.initial_modes(dev(X), dev(seeds), sigma)
    _check_assign(X, seeds, host(g_assign), o_assign)
    _check_modes(X, sigma, host(g_modes), np.array(g_dens), o_modes, o_dens, o_assign)


@pytest.mark.parametrize("N,tail", [(2100, 0), (2304, 0), (2304, 700), (5000, 0), (5000, 1500), (3000, 100),
                                    (70001, 300)])
def test_kmeanspp_largest_draw(slk, N, tail):
    """A draw just below 1 asks for the last point away from seed 0, whichever
    way the prefix sums round: never a point past the end, nor one of the `tail`
    last points, which coincide with it."""
    u = [1.0 - 2.0 ** -53]
    for seed in range(40):
        X = inputs.rng(seed).normal(size=(N, 1)).astype(np.float32)
        if tail:
            X[-tail:] = X[0]
        want = oracle.kmeanspp(X, 2, 0, u)
        assert want[1] == np.nonzero(X[:, 0] != X[0, 0])[0][-1]
        np.testing.assert_array_equal(host(slk.kmeanspp(dev(X), 2, 0, u)), want)


def test_initial_modes_distances_beyond_float32(slk):
    """Squared distances to both seeds that overflow float32 say nothing about
    the side of the border a point lies on.  Cluster 0 is its seed and a shell
    whose distances overflow; the shell's densest place is a point of cluster 1
    near its centre (every distance of that one, and their sums, are finite)."""
    U, D, n = 1e19, 64, 21000        # (enough work for the bounds to be used)
    sig = float(np.sqrt(0.72)) * U
    g = inputs.rng(17)
    shell = np.zeros((n, D))
    shell[:, 2:] = g.normal(size=(n, D - 2))
    shell *= 1.2 / np.linalg.norm(shell, axis=1, keepdims=True)
    shell[:, 1] = -0.05
    s0, s1, y = np.zeros((3, D))
    s0[:2], s1[:2], y[:2] = (1.45, -0.3), (1.45, 0.3), (0.2, 0.05)
    near1 = s1 + 0.001 * g.normal(size=(20, D))
    X = (U * np.concatenate([s0[None], s1[None], y[None], near1, shell])).astype(np.float32)
    seeds = np.array([0, 1], np.int32)
    X64 = X.astype(np.float64)
    d2 = np.stack([((X64 - X64[s]) ** 2).sum(1) for s in seeds], 1)
    top = float(np.finfo(np.float32).max)
    assert (d2[-n:] > top).all() and (d2[:-n].sum(1) < top).all()
    assign = np.where(d2[:, 0] <= d2[:, 1], 0, 1)
    assert assign[2] == 1 and (assign[-n:] == 0).all()
    sample = np.concatenate([[0, 1, 2, 3], len(X) - 1 - g.choice(n, 200, replace=False)])
    f = oracle.cluster_density(X, assign.astype(np.int32), 0, sig, sample)
    assert f.argmax() == 2 and f[2] > 2 * np.delete(f, 2).max()
    g_modes, g_assign, g_dens = slk.initial_modes(dev(X), dev(seeds), sig)
    np.testing.assert_array_equal(host(g_assign), assign)
    assert host(g_modes)[0] == 2
    assert g_dens[0] == pytest.approx(f[2], rel=DENS_RTOL)


@pytest.mark.parametrize("D", [3, 40])
def test_kmeanspp_infinite_first_seed(slk, D):
    """Seed 0 with an infinite feature: its distance to itself is not a number,
    so the first draw goes by place; its distance to seed 1 is infinite, so from
    then on no running sum exceeds u times the total and the last point is taken."""
    N = 1001
    X = inputs.rng(D).normal(size=(N, D)).astype(np.float32)
    X[5, 1] = np.inf
    got = host(slk.kmeanspp(dev(X), 4, 5, [0.25, 0.5, 0.75]))
    np.testing.assert_array_equal(got, [5, 250, N - 1, N - 1])


def _modes64(X, seeds, sigma):
    """(modes, assignment, densities) over all pairs in 64 bits."""
    Y = dev(X).double()
    assign = torch.stack([(Y - Y[int(p)]).square().sum(1) for p in seeds], 1).argmin(1)
    own = torch.nn.functional.one_hot(assign, len(seeds)).double()
    Y = Y - Y.mean(0)
    n2, f = Y.square().sum(1), []
    for a in range(0, len(X), 2048):
        d2 = (n2[a:a + 2048, None] + n2 - 2 * Y[a:a + 2048] @ Y.T).clamp_(min=0)
        f.append(torch.exp(d2.mul_(-1 / (2 * sigma * sigma))) @ own)
    dens, modes = torch.cat(f).max(0)
    return host(modes), host(assign), host(dens)


@pytest.mark.parametrize("N,D,L,sigma", [(30500, 5, 12, 0.3), (30500, 5, 12, 3.0), (30500, 5, 12, 40.0),
                                         (31001, 2, 40, 0.2), (30301, 7, 1, 1.0), (14001, 200, 7, 8.0),
                                         (30155, 16, 60, 1.0), (30140, 16, 3, 1.0)])
def test_initial_modes_other_clusters_left_out_at_size(slk, N, D, L, sigma):
    """The same at sizes from which the bounds are used (the last one is just below):
    clusters of many blocks and of less than one, ends inside a block."""
    X, _ = inputs.blobs(N=N, D=D, n_blobs=max(2, L // 2), centre_var=4.0, seed=N + L)
    seeds = inputs.kmeanspp(X, L, seed=L)
    o_modes, o_assign, o_dens = _modes64(X, seeds, sigma)
    g_modes, g_assign, g_dens = slk.initial_modes(dev(X), dev(seeds), sigma)
    _check_assign(X, seeds, host(g_assign), o_assign)
    _check_modes(X, sigma, host(g_modes), np.array(g_dens), o_modes, o_dens, o_assign)

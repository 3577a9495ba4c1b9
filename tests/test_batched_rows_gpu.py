"""The batched z-updates at the edges of their row shapes (one, two or four
labels per lane; more edges than a group has lanes; ragged last tiles) against
one solve per problem."""
import pytest

from paper_1810_13044_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def slk():
    from paper_1810_13044_gb300 import build, slk as _slk
    build.build()
    return _slk


@pytest.mark.parametrize("k", [1, 5, 24])
@pytest.mark.parametrize("affinity", ["binary", "heat"])
def test_batched_rows_equal_single(slk, k, affinity):
    probs = []
    for i, L in enumerate((1, 2, 5, 8, 9, 17, 32, 33, 64, 65, 128)):
        N = 4 * L + 261 + i
        X, _ = inputs.mixture(N, 9, max(L, 2), seed=50 + i)
        m0 = inputs.kmeanspp(X, L, seed=50 + i)
        probs.append(dict(X=torch.from_numpy(X).cuda(), L=L, k=k, lam=0.7,
                          init_modes=torch.from_numpy(m0).cuda()))
    p = slk.default_params(affinity=affinity)
    for pr, (Z, lab, modes, st) in zip(probs, slk.solve_batched(probs, params=p)):
        Z1, lab1, modes1, st1 = slk.solve(pr["X"], pr["L"], k, pr["lam"], pr["init_modes"], params=p)
        assert st["outer_iters"] == st1["outer_iters"]
        assert st["inner_iters_total"] == st1["inner_iters_total"]
        assert torch.equal(modes, modes1) and torch.equal(lab, lab1)
        assert (Z - Z1).abs().max().item() <= 1e-6

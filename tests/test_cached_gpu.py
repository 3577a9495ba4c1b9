"""The cached z-updates on both sides of the line between their two tilings (two
labels per lane), against the oracle."""
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


def _line(lanes, k):
    """The largest N of the small-problem tiling, `lanes` lanes per row."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152
    return (210 if k <= 5 else 77) * 4 * 256 * sms // (100 * lanes)


@pytest.mark.parametrize("L,lanes", [(9, 8), (16, 8), (17, 16), (32, 16), (33, 32), (64, 32)])
@pytest.mark.parametrize("k", [1, 5, 6])
@pytest.mark.parametrize("side", [0, 1])
def test_small_and_large_problems(slk, L, lanes, k, side):
    N = _line(lanes, k) + side
    rp, ci, w = inputs.random_graph(N, k, seed=N, weighted=bool(k % 2))
    A = inputs.random_unary(N, L, seed=L)
    Z0 = inputs.random_simplex_rows(N, L, seed=L + 1)
    d = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()
    Z, Zp = d(Z0), torch.empty(N, L, device="cuda")
    it, _ = slk.bound_iterate(d(A), d(rp), d(ci), d(w), 0.8, Z, Zp, 3, tol=-1.0)
    Zo, Zpo, _, _ = oracle.bound_iterate(A, rp, ci, w, 0.8, Z0, 3)
    assert it == 3
    assert np.abs(Z.cpu().numpy() - Zo).max() <= Z_TOL
    assert np.abs(Zp.cpu().numpy() - Zpo).max() <= Z_TOL

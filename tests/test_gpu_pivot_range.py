"""Mixed precision at the ends of the FP32 range: pivots that are subnormal, or
whose reciprocal is, on every tiling."""
import numpy as np
import pytest

from paper_2403_16341_gb300 import inputs as I
from tests.parity import gpu_solve

pytestmark = pytest.mark.gpu

NEWTON = 0
MIXED, TILE_THREAD, TILE_WARP, TILE_CTA, REFINE = 1 << 8, 1 << 10, 1 << 11, 1 << 12, 1 << 14


@pytest.fixture(scope="module")
def solver():
    import paper_2403_16341_gb300 as nls
    s = nls.Solver(0)
    yield s
    s.close()


@pytest.mark.parametrize("n,tiling", [(8, TILE_THREAD), (8, TILE_WARP), (16, TILE_WARP), (31, TILE_WARP), (8, TILE_CTA),
                                      (16, TILE_CTA), (40, TILE_CTA), (128, TILE_CTA)])
@pytest.mark.parametrize("pivot", [1e-38, 2.0 ** -126, 2.0 ** 126, 1.5e38, 3e38])
def test_one_newton_step_with_extreme_pivots(solver, n, tiling, pivot):
    # diagonal cubic systems at u0 = 0: J = A, so one Newton step is u_i = b_i / A_ii.
    # A, b and the product round (1.4e-7 at most each, subnormal ones among them: no
    # more than two of the three here), the approximate reciprocal is off by 1.2e-7
    # and rounds to a subnormal number (2.1e-7 for a pivot of 3e38): below 6e-7.
    B = 5
    rng = np.random.default_rng(n)
    A = np.zeros((n, n, B))
    d = np.where(rng.random((n, B)) < 0.5, pivot, 3.0) * rng.choice([-1.0, 1.0], (n, B))
    A[np.arange(n), np.arange(n)] = d
    want = rng.uniform(0.5, 1.0, (n, B))
    b = I.Batch(I.FAMILY_CUBIC, n, np.concatenate([A.reshape(n * n, B), d * want]), np.zeros((n, B)))
    g = gpu_solve(solver, b, NEWTON | MIXED | tiling, abstol=0.0, maxiters=1)
    assert np.abs(g["u"] / want - 1.0).max() < 6e-7

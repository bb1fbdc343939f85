"""The FP64 reciprocal over its whole range: at u0 = 0 a cubic system of n = 1 with
b = 1 takes the step 1 / A exactly (the step is 1 times the reciprocal)."""
import numpy as np
import pytest

from paper_2403_16341_gb300 import inputs as I
from tests.parity import gpu_solve

pytestmark = pytest.mark.gpu

NEWTON = 0
TILE_THREAD, TILE_WARP, TILE_CTA = 1 << 10, 1 << 11, 1 << 12


@pytest.mark.parametrize("tiling", [TILE_THREAD, TILE_WARP, TILE_CTA])
def test_reciprocal_of_every_exponent(tiling):
    import paper_2403_16341_gb300 as nls
    rng = np.random.default_rng(5)
    e = np.repeat(np.arange(-1022, 1024), 4)
    m = np.concatenate([rng.uniform(1.0, 2.0, e.size - 6), [1.0, 2.0 - 2.0 ** -52, 1.0 + 2.0 ** -52] * 2])
    A = np.ldexp(m, np.concatenate([e[:-6], [-1022] * 3, [1023] * 3]))
    sub = np.ldexp(rng.uniform(1.0, 2.0, 200), rng.integers(-1074, -1022, 200))  # subnormal: some reciprocals overflow
    A = np.concatenate([A, sub[sub > 0], np.ldexp(1.0, np.arange(-1074, 1024))])
    A *= rng.choice([-1.0, 1.0], A.size)
    s = nls.Solver(0)
    g = gpu_solve(s, I.Batch(I.FAMILY_CUBIC, 1, np.stack([A, np.ones_like(A)]), np.zeros((1, A.size))), NEWTON | tiling,
                  abstol=0.0, maxiters=1)
    s.close()
    with np.errstate(over="ignore"):
        want = 1.0 / A
    np.testing.assert_array_equal(g["u"][0], want)

"""Persistent grids of several waves, where instances are drawn from the work
counter and idle lanes refilled, against static grids: the same bits on every
tiling and at every refill threshold, the unset default among them."""
import numpy as np
import pytest

from paper_2403_16341_gb300 import inputs as I
from tests.parity import gpu_solve

pytestmark = pytest.mark.gpu

NEWTON, LS, TR, POTRA = 0, 1, 2, 4
MIXED, TILE_WARP = 1 << 8, 1 << 11


def solved(b, alg, **options):
    import paper_2403_16341_gb300 as nls
    s = nls.Solver(0)  # every option at its default
    s.set_option(nls.NLS_OPT_CTAS_PER_SM, 1)
    for name, value in options.items():
        s.set_option(getattr(nls, "NLS_OPT_" + name), value)
    g = gpu_solve(s, b, alg)
    s.close()
    return g


def same(a, g):
    for key in ("u", "status", "iters", "resid", "nfev", "solved"):
        np.testing.assert_array_equal(a[key], g[key], err_msg=key)


@pytest.mark.parametrize("family,n,alg", [("cubic", 8, LS), ("cubic", 8, TR | MIXED), ("cubic", 3, NEWTON), ("bratu", 5, TR),
                                          ("rosenbrock", 6, TR), ("cubic", 8, POTRA)])
def test_thread_tiling_refills(family, n, alg):
    B = 15013  # 470 warps, three waves at one CTA of a warp per SM
    b = {"cubic": I.cubic_batch, "bratu": I.bratu_batch, "rosenbrock": I.rosenbrock_batch}[family](n, B, config_id=7)
    want = solved(b, alg, PERSISTENT=0)
    same(want, solved(b, alg))
    for refill in (0, 8, 24, 31):
        same(want, solved(b, alg, REFILL_BELOW=refill))


@pytest.mark.parametrize("family,n,alg,B", [("cubic", 12, TR, 3001), ("bratu", 16, LS | MIXED, 3001), ("cubic", 32, LS | MIXED, 901),
                                            ("cubic", 27, TR, 901), ("square", 8, LS | TILE_WARP, 5003), ("cubic", 40, TR, 401),
                                            ("bratu", 40, TR | MIXED, 401), ("bratu", 65, LS | MIXED, 401),
                                            ("bratu", 48, TR | MIXED, 1301)])
def test_warp_and_cta_tilings_draw(family, n, alg, B):
    b = {"cubic": I.cubic_batch, "bratu": I.bratu_batch, "square": I.square_batch}[family](n, B, config_id=7)
    same(solved(b, alg, PERSISTENT=0), solved(b, alg))

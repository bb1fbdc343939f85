"""The warp- and CTA-tiled LU at the edges of their tiles, panels and chunks,
on systems that interchange rows at nearly every step and hold equal pivot
candidates; the FP64 reciprocal; the request counters over more than one lap
of their ring."""
import numpy as np
import pytest

from paper_2403_16341_gb300 import inputs as I
from tests.parity import check_parity, gpu_solve, oracle_solve

pytestmark = pytest.mark.gpu

NEWTON, LS, TR, HALLEY = 0, 1, 2, 5
MIXED, TILE_WARP, TILE_CTA, REFINE = 1 << 8, 1 << 11, 1 << 12, 1 << 14


@pytest.fixture(scope="module")
def solver():
    import paper_2403_16341_gb300 as nls
    s = nls.Solver(0)
    yield s
    s.close()


def interchanging(n, B, ties):
    """Cubic systems whose rows are shuffled, so that the largest entry of a
    column is rarely on the diagonal; with `ties`, G takes the values -1/8, 0
    and 1/8 only, so that many candidates are equal.  b is small: the systems
    are close to linear and Newton's path is short."""
    b = I.cubic_batch(n, B, config_id=7, b_half_width=0.1)
    A = b.params[: n * n].reshape(n, n, B)
    if ties:
        G = A - 3.0 * np.eye(n)[:, :, None]
        A[:] = 3.0 * np.eye(n)[:, :, None] + np.clip(np.rint(2.0 * G / max(I.cubic_g_sigma(n), 1e-3)), -1, 1) / (8 * n ** 0.5)
    rng = np.random.default_rng(n)
    for k in range(B):
        A[:, :, k] = A[rng.permutation(n), :, k]
    return b


@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("alg", [LS, TR, LS | MIXED, TR | MIXED])
@pytest.mark.parametrize("n", [2, 8, 9, 16, 17, 31, 32])
def test_warp_lu_interchanges(solver, n, alg, ties):
    b = interchanging(n, 37, ties)
    g = gpu_solve(solver, b, alg | TILE_WARP)
    check_parity(b, g, oracle_solve(b, alg & 3), bool(alg & MIXED))


@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("alg", [LS, TR, LS | MIXED, TR | MIXED, TR | MIXED | REFINE])
@pytest.mark.parametrize("n", [1, 4, 5, 8, 31, 33, 40, 41, 63, 64, 65, 96, 97, 127, 128])
def test_cta_lu_interchanges(solver, n, alg, ties):
    b = interchanging(n, 7, ties)
    g = gpu_solve(solver, b, alg | TILE_CTA)
    check_parity(b, g, oracle_solve(b, alg & 3), bool(alg & MIXED))


@pytest.mark.parametrize("alg", [LS, LS | MIXED, LS | MIXED | REFINE])
@pytest.mark.parametrize("n", [33, 128])
def test_cta_singular_and_nan_instances_leave_the_others(solver, n, alg):
    import oracle as O
    b = interchanging(n, 6, False)
    A = b.params[: n * n].reshape(n, n, 6)
    A[:, n - 1, 1] = 0.0  # a zero column at u0 = 0: singular in the last panel
    A[n // 2, 0, 4] = np.inf  # F(u0) = Inf * 0 is NaN
    g = gpu_solve(solver, b, alg | TILE_CTA)
    assert g["status"][1] == O.ST_SINGULAR and g["status"][4] == O.ST_NONFINITE
    assert (np.delete(g["status"], [1, 4]) == 0).all()


def test_fp64_reciprocal_is_correctly_rounded(solver):
    # one Newton pass on u^2 = p, n = 1: u1 = u0 + (-F) * RN(1 / (2 u0)), so the
    # exact bits follow from IEEE arithmetic (the compiler may fuse the last
    # multiply and add: either rounding is right)
    rng = np.random.default_rng(3)
    m = np.concatenate([rng.uniform(1.0, 2.0, 40000), 1.0 + np.arange(64) * 2.0 ** -52, 2.0 - np.arange(1, 65) * 2.0 ** -53])
    u0 = np.ldexp(m, rng.integers(-400, 400, m.size)) * rng.choice([-1.0, 1.0], m.size)
    p = u0 * u0 * rng.uniform(0.5, 2.0, m.size)
    b = I.Batch(I.FAMILY_SQUARE, 1, p[None].copy(), u0[None].copy())
    g = gpu_solve(solver, b, NEWTON, abstol=0.0, maxiters=1)
    from fractions import Fraction
    for k in list(range(0, m.size, 211)) + list(range(m.size - 128, m.size)):
        F = float(Fraction(u0[k]) * Fraction(u0[k]) - Fraction(p[k]))  # one fused operation
        r = 1.0 / (2.0 * u0[k])
        want = (u0[k] + (-F) * r, float(Fraction(-F) * Fraction(r) + Fraction(u0[k])))
        assert g["u"][0, k] in want, (k, u0[k].hex(), g["u"][0, k].hex(), [w.hex() for w in want])


def test_counters_over_two_laps_of_the_ring(solver):
    # 2 of the 65,536 ring entries per request; some requests are collected only
    # after their entries were reused
    import torch

    import paper_2403_16341_gb300 as nls
    b = I.square_batch(2, 5)
    p, u0 = torch.from_numpy(b.params).cuda(), torch.from_numpy(b.u0).cuda()
    u = torch.empty_like(u0)
    early = []
    for i in range(34000):
        if i % 5000 < 2:  # every launch solves from u0 or meets the roots: 5 solved
            u.copy_(u0)
        r = solver.submit(nls.NLS_SQUARE, p, u, NEWTON)
        solver.flush()
        if i in (3, 4, 9000):
            early.append(r)
        elif i % 64 == 63 or i > 33000:
            assert solver.wait(r) == 5
        else:
            early.append(r) if i % 1000 == 0 else solver.wait(r)
    assert [solver.wait(r) for r in early] == [5] * len(early)
    # several requests in one flush on the second lap
    us = [u0.clone() for _ in range(4)]
    reqs = [solver.submit(nls.NLS_SQUARE, p, v, NEWTON) for v in us]
    solver.flush()
    assert [solver.wait(r) for r in reqs] == [5] * 4

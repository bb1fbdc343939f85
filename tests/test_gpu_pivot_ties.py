"""Equal pivot candidates: the lowest position among equals is taken, and FP64
candidates whose high words are equal are told apart by their low words.

A pair of equations (1, M), (1, 1) in two unknowns, M = 2^60, right-hand sides
M and 3, shows which row was the pivot: with the first, 1 - M and 3 - M lose the
small terms and the first unknown is not 2; with the second it is.  At u0 = 0 the
cubic family's Jacobian is A, so one Newton step returns that solution."""
import numpy as np
import pytest

from paper_2403_16341_gb300 import inputs as I
from tests.parity import gpu_solve

pytestmark = pytest.mark.gpu

NEWTON = 0
MIXED, TILE_WARP, TILE_CTA = 1 << 8, 1 << 11, 1 << 12
M = 2.0 ** 60


@pytest.fixture(scope="module")
def solver():
    import paper_2403_16341_gb300 as nls
    s = nls.Solver(0)
    yield s
    s.close()


def paired(n, B, low_words):
    """B systems of n // 2 pairs in random rows and columns (an odd n: one row more
    of its own).  low_words: the two candidates differ in the last bits only."""
    rng = np.random.default_rng(100 * n + low_words)
    A, b = np.zeros((n, n, B)), np.zeros((n, B))
    for k in range(B):
        rows, cols = rng.permutation(n), rng.permutation(n)
        for q in range(n // 2):
            (i, j), (c, d) = rows[2 * q: 2 * q + 2], sorted(cols[2 * q: 2 * q + 2])
            s = rng.choice([-1.0, 1.0], 2)  # whole rows change sign
            A[i, c, k], A[i, d, k], b[i, k] = s[0], s[0] * M, s[0] * M
            A[j, c, k], A[j, d, k], b[j, k] = s[1], s[1], s[1] * 3.0
            if low_words:
                A[(i, j)[rng.integers(2)], c, k] *= 1.0 + 2.0 ** -50
        if n % 2:
            A[rows[-1], cols[-1], k], b[rows[-1], k] = 1.0, 1.0
    return A, b


def pivots(A):
    """Row of A that each step of the LU takes, and how many steps met equal candidates."""
    a, pos, ties, out = A.copy(), np.arange(len(A)), 0, []
    n = len(A)
    order = np.arange(n)  # row at each position
    for k in range(n):
        m = np.abs(a[order[k:], k])
        p = k + int(np.argmax(m))  # the first of the largest
        ties += int((m == m.max()).sum() > 1)
        order[[k, p]] = order[[p, k]]
        r = order[k]
        out.append(r)
        for i in order[k + 1:]:
            if a[i, k]:
                a[i, k + 1:] -= a[i, k] / a[r, k] * a[r, k + 1:]
    return out, ties


@pytest.mark.parametrize("low_words", [False, True])
@pytest.mark.parametrize("n,tiling,many", [(2, TILE_WARP, 0), (8, TILE_WARP, 0), (9, TILE_WARP, 0), (16, TILE_WARP, 0),
                                           (17, TILE_WARP, 0), (31, TILE_WARP, 0), (32, TILE_WARP, 0), (2, TILE_CTA, 0),
                                           (9, TILE_CTA, 0), (33, TILE_CTA, 0), (64, TILE_CTA, 0), (65, TILE_CTA, 0),
                                           (96, TILE_CTA, 0), (127, TILE_CTA, 0), (128, TILE_CTA, 0), (9, TILE_CTA, 1),
                                           (33, TILE_CTA, 1), (64, TILE_CTA, 1), (96, TILE_CTA, 1)])
@pytest.mark.parametrize("mixed", [0, MIXED])
def test_pivot_among_equals(solver, n, tiling, many, low_words, mixed):
    # many: more instances than the mixed kernel of small batches takes
    if mixed and low_words:
        pytest.skip("an FP32 entry has one word")
    if many and not mixed:
        pytest.skip("one FP64 kernel serves all batches")
    B = 7
    A, b = paired(n, B, low_words)
    reps = (3200 if n <= 64 else 700) // B if many else 1
    g = gpu_solve(solver, I.Batch(I.FAMILY_CUBIC, n, np.tile(np.concatenate([A.reshape(n * n, B), b]), (1, reps)),
                                  np.zeros((n, B * reps))), NEWTON | mixed | tiling, abstol=0.0, maxiters=1)
    ties = 0
    for k in range(B):
        order, t = pivots(A[:, :, k])
        ties += t
        for c in range(n):
            r = order[c]  # the pivot row of column c
            if (A[:, c, k] != 0).sum() != 2 or np.abs(A[r, :, k]).max() not in (M, 1.0, 1.0 + 2.0 ** -50):
                continue
            if np.abs(A[:, c, k]).max() > 1.5:
                continue  # the pair's second column
            first = np.abs(A[r, :, k]).max() == M  # the row (1, M) was the pivot
            other = np.flatnonzero(A[r, :, k])
            if len(other) != 2 or other[0] != c:
                continue
            for i in range(reps):
                x = g["u"][c, k + i * B]
                assert (abs(x - 2.0) > 0.5) == first, (k, c, x)
    assert low_words or ties > B * (n // 2) // 2

"""The two mixed-precision kernels of the CTA tiling: batches up to one wave (the
cubic: more) run on the register panels, larger ones on the shared-memory
columns; an instance gets the same bits on both."""
import numpy as np
import pytest

from paper_2403_16341_gb300 import inputs as I
from tests.parity import gpu_solve
from tests.test_gpu_lu_edges import interchanging

pytestmark = pytest.mark.gpu

NEWTON, LS, TR = 0, 1, 2
MIXED, TILE_CTA, REFINE = 1 << 8, 1 << 12, 1 << 14
MOST = 20  # instances per SM: above five waves of four CTAs no family stays on the panels


@pytest.fixture(scope="module")
def solver():
    import paper_2403_16341_gb300 as nls
    s = nls.Solver(0)
    yield s
    s.close()


def repeated(b, B):
    k = np.arange(B) % b.batch
    return I.Batch(b.family, b.n, np.ascontiguousarray(b.params[:, k]), np.ascontiguousarray(b.u0[:, k]))


def batch(family, n):
    if family == "cubic":
        return interchanging(n, 7, n % 2 == 0)
    if family == "bratu":
        return I.bratu_batch(n, 7, config_id=7)
    if family == "square":
        return I.square_batch(n, 7)
    return I.rosenbrock_batch(n, 7)


@pytest.mark.parametrize("n", [1, 4, 31, 33, 40, 41, 63, 64, 65, 95, 96, 97])
@pytest.mark.parametrize("family", ["cubic", "bratu", "square", "rosenbrock"])
def test_small_and_large_batches_give_the_same_bits(solver, family, n):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    small = batch(family, n)
    large = repeated(small, (MOST if family == "cubic" and n <= 64 else 4) * sms + 1)
    for alg in (NEWTON, LS, TR, TR | REFINE):
        a = gpu_solve(solver, small, alg | MIXED | TILE_CTA)
        g = gpu_solve(solver, large, alg | MIXED | TILE_CTA)
        k = np.arange(large.batch) % small.batch
        for key in ("u", "status", "iters", "nfev", "resid"):
            np.testing.assert_array_equal(g[key], a[key][..., k], err_msg=f"{key}, alg {alg}")


def test_the_instances_of_a_flush_decide_together(solver):
    # 40 requests that would each run on the panels, one flush: the same bits
    import torch
    held, reqs = [], []
    for i in range(40):
        b = repeated(batch(("cubic", "bratu")[i % 2], 48), 100)
        p, u = torch.from_numpy(b.params).cuda(), torch.from_numpy(b.u0).cuda()
        held.append((b, p, u))
        reqs.append(solver.submit(b.family, p, u, TR | MIXED, 1e-10, 50))
    solver.flush()
    solved = [solver.wait(r) for r in reqs]
    for (b, p, u), s in zip(held[:2], solved[:2]):
        a = gpu_solve(solver, b, TR | MIXED)
        np.testing.assert_array_equal(u.cpu().numpy(), a["u"])
        assert s == a["solved"]
    for i, (b, p, u) in enumerate(held):
        assert torch.equal(u, held[i % 2][2]) and solved[i] == solved[i % 2]

"""The ring of request counters on the GPU: flushes that take entries zeroed on
another stream, reuse of entries that kernels wrote."""
import numpy as np
import pytest

from paper_2403_16341_gb300 import inputs as I

pytestmark = pytest.mark.gpu

NEWTON = 0
ENTRIES = 2  # of the ring, per request
BLOCK = 1 << 12  # entries zeroed at a time


@pytest.fixture()
def solver():
    import paper_2403_16341_gb300 as nls
    s = nls.Solver(0)  # a ring of its own
    yield s
    s.close()


def on_gpu(b):
    import torch
    return torch.from_numpy(np.ascontiguousarray(b.params)).cuda(), torch.from_numpy(np.ascontiguousarray(b.u0)).cuda()


def test_rest_of_a_block_zeroed_on_the_second_solve_stream(solver):
    # a host request of 2^18 instances in flight, its second chunk (on the second
    # solve stream) the one that crosses into a block of the ring; then 2,100
    # requests in one flush on the handle's stream
    import torch

    import paper_2403_16341_gb300 as nls
    b = I.square_batch(2, 5)
    p, u0 = on_gpu(b)
    u = u0.clone()
    for _ in range(BLOCK // ENTRIES - 1):
        r = solver.submit(nls.NLS_SQUARE, p, u, NEWTON)
        solver.flush()
        solver.wait(r)
    big = I.square_batch(2, 1 << 18)
    hu = big.u0.copy()
    hreq = nls.nls_solve_host_async(solver.h, big.family, big.params.ctypes.data, hu.ctypes.data, big.n, big.batch,
                                    NEWTON, 1e-10, 50)
    us = [u0.clone() for _ in range(2100)]
    reqs = [solver.submit(nls.NLS_SQUARE, p, v, NEWTON) for v in us]
    solver.flush()
    assert [solver.wait(r) for r in reqs] == [b.batch] * len(us)
    assert nls.nls_status(solver.h, hreq) == big.batch
    want = np.sqrt(b.params)
    assert np.abs(torch.stack(us).cpu().numpy() - want).max() < 1e-9
    assert np.abs(hu - np.sqrt(big.params)).max() < 1e-9


@pytest.mark.parametrize("lone", [True, False])
def test_captured_flush_replays_beside_direct_ones(lone):
    # a flush recorded by a stream capture: each replay solves from the u at that
    # time; direct flushes between replays, through a whole lap of the ring, are
    # right as well
    import torch

    import paper_2403_16341_gb300 as nls
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        solver = nls.Solver(0)
        solver.set_option(nls.NLS_OPT_CTAS_PER_SM, 1)
        b = I.square_batch(2, 40000)  # several waves: a work counter
        p, u0 = on_gpu(b)
        groups = [u0.clone() for _ in range(1 if lone else 3)]
        stat = torch.empty(b.batch, dtype=torch.int32, device="cuda")
        small = I.square_batch(2, 5)
        sp, su0 = on_gpu(small)
        su = su0.clone()

        def direct():
            su.copy_(su0)
            r = solver.submit(nls.NLS_SQUARE, sp, su, NEWTON)
            solver.flush()
            assert solver.wait(r) == small.batch

        direct()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            for v in groups:
                solver.submit(nls.NLS_SQUARE, p, v, NEWTON, 1e-10, 50, (stat, None, None, None))
            solver.flush()
        want = np.sqrt(b.params)

        def replay():
            for v in groups:
                v.copy_(u0)
            stat.fill_(-1)
            g.replay()
            st.synchronize()
            for v in groups:
                assert np.abs(v.cpu().numpy() - want).max() < 1e-9
            assert (stat == 0).all()

        for _ in range(3):
            replay()
            direct()
        big = u0.clone()
        for i in range((1 << 16) // ENTRIES + 8):
            if i % 4096 == 0:
                replay()
                big.copy_(u0)
                r = solver.submit(nls.NLS_SQUARE, p, big, NEWTON)
                solver.flush()
                assert solver.wait(r) == b.batch
                assert np.abs(big.cpu().numpy() - want).max() < 1e-9
            else:
                direct()
        replay()
        st.synchronize()
        solver.close()


def test_entries_are_zero_again_on_the_second_lap(solver):
    # two laps of the same layout: groups, lone requests of several waves (whose
    # work counters end above their batch) and now and then a host request on
    # both solve streams; a counter that is not zeroed again would have the
    # grids of the second lap skip their instances
    import paper_2403_16341_gb300 as nls
    solver.set_option(nls.NLS_OPT_CTAS_PER_SM, 1)
    small, waves, big = I.square_batch(2, 5), I.square_batch(2, 6000), I.square_batch(2, 1 << 18)
    sp, su0 = on_gpu(small)
    wp, wu0 = on_gpu(waves)
    us = [su0.clone() for _ in range(500)]
    wu = wu0.clone()
    want, want_host = np.sqrt(waves.params), np.sqrt(big.params)
    for lap in range(2):
        for turn in range(64):
            for v in us:
                v.copy_(su0)
            reqs = [solver.submit(nls.NLS_SQUARE, sp, v, NEWTON) for v in us[: 500 - 2 * (turn % 16 == 5)]]
            solver.flush()
            if turn % 16 == 5:
                hu = big.u0.copy()
                nls.nls_solve_host(solver.h, big.family, big.params.ctypes.data, hu.ctypes.data, big.n, big.batch, NEWTON,
                                   1e-10, 50)
                assert np.abs(hu - want_host).max() < 1e-9
            for _ in range(12):
                wu.copy_(wu0)
                r = solver.submit(nls.NLS_SQUARE, wp, wu, NEWTON)
                solver.flush()
                assert solver.wait(r) == waves.batch, (lap, turn)
            assert np.abs(wu.cpu().numpy() - want).max() < 1e-9
            assert [solver.wait(r) for r in reqs] == [small.batch] * len(reqs), (lap, turn)

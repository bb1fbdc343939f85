"""The solved count of a lone request on both sides of the switch from adds into
pinned memory to a copy behind the kernel, on every tiling."""
import pytest

from paper_2403_16341_gb300 import inputs as I

pytestmark = pytest.mark.gpu

NEWTON = 0
TILE_THREAD, TILE_WARP, TILE_CTA = 1 << 10, 1 << 11, 1 << 12


@pytest.mark.parametrize("n,tiling,batches", [(4, TILE_THREAD, (1, 4096 * 32, 4096 * 32 + 1)),
                                              (8, TILE_WARP, (2048, 2049, 5000)), (16, TILE_WARP, (1023, 1024, 1025, 4096)),
                                              (32, TILE_WARP, (511, 512, 513)), (40, TILE_CTA, (1, 511, 512, 513, 1000))])
def test_solved_count_of_lone_requests(n, tiling, batches):
    import torch

    import paper_2403_16341_gb300 as nls
    s = nls.Solver(0)
    for persistent in (1, 0):
        s.set_option(nls.NLS_OPT_PERSISTENT, persistent)
        for B in batches:
            b = I.square_batch(n, B)
            b.params[0, B // 2] = -1.0  # no root: this instance is not counted
            p, u = torch.from_numpy(b.params).cuda(), torch.from_numpy(b.u0).cuda()
            for _ in range(2):
                v = u.clone()
                r = s.submit(b.family, p, v, NEWTON | tiling)
                s.flush()
                assert s.wait(r) == B - 1
    s.close()

"""Masks without any background: every distance is 0xFFFFFFFF and every site -1,
whatever the context transformed before, and no row or column is searched for
nothing."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1311_0378_gb300 as rc  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    import paper_1311_0378_gb300.build as b
    b.build()
    c = rc.recon_init(0, 0, rc.RECON_FLAG_SYNC)
    yield c
    rc.recon_free(c)


def transform(ctx, B, with_site):
    d2 = torch.zeros(B.shape, dtype=torch.int32, device="cuda")
    site = torch.zeros_like(d2)
    torch.cuda.synchronize()
    rc.check(rc.recon_dt(ctx, B.data_ptr(), d2.data_ptr(), site.data_ptr() if with_site else 0, *B.shape))
    return d2.cpu().numpy().view(np.uint32), site.cpu().numpy()


# (columns of more than 8192 rows are looked at first; 32767 rows up is the largest distance)
@pytest.mark.parametrize("shape", [(1, 1), (1, 515), (33, 1), (32, 512), (65, 1027), (3, 9001), (300, 700), (20000, 7),
                                   (32768, 2)])
def test_with_and_without_background_in_turn(ctx, shape):
    full = torch.ones(shape, dtype=torch.uint8, device="cuda")
    for y, x in ((0, 0), (shape[0] - 1, shape[1] - 1)):
        one = full.clone()
        one[y, x] = 0
        yy, xx = np.mgrid[0:shape[0], 0:shape[1]]
        for with_site in (False, True):
            d2, site = transform(ctx, full, with_site)
            assert (d2 == 0xFFFFFFFF).all() and (site == (-1 if with_site else 0)).all()
            d2, site = transform(ctx, one, with_site)
            np.testing.assert_array_equal(d2, (yy - y) ** 2 + (xx - x) ** 2)
            assert (site == (y * shape[1] + x if with_site else 0)).all()


def test_costs_no_more_than_a_mask_with_background(ctx):
    """The work without background is a part of that with some (reading the mask,
    writing the results); a search from end to end of every row takes 20 times it."""
    full = torch.ones((4096, 4096), dtype=torch.uint8, device="cuda")
    some = (torch.rand((4096, 4096), device="cuda") < 0.99).to(torch.uint8)
    d2 = torch.empty((4096, 4096), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()

    def best(B):
        out = []
        for _ in range(12):
            t = time.perf_counter()
            rc.check(rc.recon_dt(ctx, B.data_ptr(), d2.data_ptr(), 0, 4096, 4096))
            out.append(time.perf_counter() - t)
        return min(out)
    assert best(full) <= 3 * best(some)

"""The distance transform is exact and takes the site with the lowest index
among the nearest: sizes around its 32-row strips and 32-column runs, rows too
wide for the default shared memory, columns and rows without background. Whole
numbers, so the tolerance is zero."""
import numpy as np
import pytest
from scipy import ndimage

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1311_0378_gb300 as rc  # noqa: E402


def gpu_dt(B, want_site, lead=0):
    import paper_1311_0378_gb300.build as b
    b.build()
    H, W = B.shape
    buf = torch.zeros(lead + H * W, dtype=torch.uint8, device="cuda")
    buf[lead:] = torch.from_numpy(np.ascontiguousarray(B)).cuda().view(-1)
    d2 = torch.empty((H, W), dtype=torch.int32, device="cuda")
    site = torch.empty((H, W), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    c = rc.recon_init(0, 0, rc.RECON_FLAG_SYNC)
    try:
        rc.check(rc.recon_dt(c, buf.data_ptr() + lead, d2.data_ptr(), site.data_ptr() if want_site else 0, H, W))
    finally:
        rc.recon_free(c)
    return site.cpu().numpy(), d2.cpu().numpy().view(np.uint32).astype(np.int64)


def exact(B):
    H, W = B.shape
    i = ndimage.distance_transform_edt(B, return_distances=False, return_indices=True)
    y, x = np.mgrid[0:H, 0:W]
    return (i[0] - y) ** 2 + (i[1] - x) ** 2


def lowest_site(B):
    ys, xs = np.nonzero(B == 0)
    H, W = B.shape
    y, x = np.mgrid[0:H, 0:W]
    d = (y[..., None] - ys) ** 2 + (x[..., None] - xs) ** 2
    return (ys * W + xs)[np.argmin(d, axis=-1)]   # nonzero() lists by index: argmin takes the lowest


@pytest.mark.parametrize("shape", [(1, 1), (1, 40), (40, 1), (31, 33), (32, 32), (33, 31), (65, 70), (97, 130)])
@pytest.mark.parametrize("density", [0.5, 0.9, 0.99, 0.999])
def test_small(shape, density):
    rng = np.random.default_rng(int(1000 * density) + shape[0] * 7 + shape[1])
    B = (rng.random(shape) < density).astype(np.uint8)
    B[rng.integers(shape[0]), rng.integers(shape[1])] = 0
    want_site = lowest_site(B)
    for lead in (0, 1):
        site, d2 = gpu_dt(B, True, lead)
        np.testing.assert_array_equal(d2, exact(B))
        np.testing.assert_array_equal(site, want_site)
        np.testing.assert_array_equal(gpu_dt(B, False, lead)[1], d2)


@pytest.mark.parametrize("shape,sites", [((300, 9001), 3), ((1200, 700), 1), ((64, 20000), 40), ((3000, 64), 2),
                                         ((777, 1031), 200)])
def test_far_sites(shape, sites):
    rng = np.random.default_rng(shape[1] + sites)
    B = np.ones(shape, np.uint8)
    B[rng.integers(shape[0], size=sites), rng.integers(shape[1], size=sites)] = 0
    site, d2 = gpu_dt(B, True)
    np.testing.assert_array_equal(d2, exact(B))
    y, x = np.mgrid[0:shape[0], 0:shape[1]]
    assert (B.reshape(-1)[site] == 0).all()
    np.testing.assert_array_equal((y - site // shape[1]) ** 2 + (x - site % shape[1]) ** 2, d2)
    np.testing.assert_array_equal(gpu_dt(B, False)[1], d2)

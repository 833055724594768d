"""GPU: the distance transform's row skipping and its four-pixel initialisation at the edges:
widths on both sides of a multiple of 4 and of the 64-column tile, arrays that are not aligned for
the wide accesses, rows without foreground between rows with it, runs of rows."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1605_00930_gb300 import iwpp
from tests._edt_checks import check_valid, exact_d2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [4, 62, 63, 64, 68, 129])
@pytest.mark.parametrize("conn", [4, 8])
def test_layouts(W, conn):
    rng = np.random.default_rng([W, conn])
    for H in (3, 16, 35):
        fg = (rng.random((H, W)) < 0.9).astype(np.uint8)
        fg[rng.random(H) < 0.4] = 0   # rows of background only
        fg[0, 0] = 0
        for off in (0, 1):            # mask off by a byte, outputs by a word
            m = torch.zeros(H * W + 16, dtype=torch.uint8, device="cuda")[off:off + H * W].view(H, W)
            m.copy_(torch.from_numpy(fg))
            site = torch.empty(H * W + 4, dtype=torch.int32, device="cuda")[off:off + H * W].view(H, W)
            d2 = torch.empty(H * W + 4, dtype=torch.int32, device="cuda")[off:off + H * W].view(H, W)
            T = iwpp.DistanceTransform(H, W)
            assert T(m, site, d2, conn) == 0 and T.status() == 0
            s, d = site.cpu().numpy().view(np.uint32).astype(np.int64), d2.cpu().numpy().astype(np.int64)
            check_valid(fg, s >> 16, s & 0xFFFF, d, conn)
            assert np.all(d >= exact_d2(fg))
            site2 = torch.empty_like(site)
            assert T(m, site2, None, conn) == 0 and T.status() == 0   # without the distances
            s2 = site2.cpu().numpy().view(np.uint32).astype(np.int64)
            yy, xx = np.mgrid[0:H, 0:W]
            check_valid(fg, s2 >> 16, s2 & 0xFFFF, (yy - (s2 >> 16)) ** 2 + (xx - (s2 & 0xFFFF)) ** 2, conn)


@pytest.mark.parametrize("H,W", [(1, 4000), (4000, 1), (700, 66), (66, 700), (333, 335)])
@pytest.mark.parametrize("conn", [4, 8])
def test_one_site_travels_through_every_tile(H, W, conn):
    # rows of a tile that follow one another are one run, from above and from below; one site is exact
    for y, x in ((0, 0), (H - 1, W - 1), (H // 2, W // 2)):
        fg = np.ones((H, W), np.uint8)
        fg[y, x] = 0
        d2 = torch.empty((H, W), dtype=torch.int32, device="cuda")
        T = iwpp.DistanceTransform(H, W)
        assert T(torch.from_numpy(fg).cuda(), torch.empty_like(d2), d2, conn) == 0 and T.status() == 0
        yy, xx = np.mgrid[0:H, 0:W]
        assert np.array_equal(d2.cpu().numpy(), (yy - y) ** 2 + (xx - x) ** 2)


@pytest.mark.parametrize("H,W", [(1, 1), (16, 64), (37, 201), (200, 333)])
def test_distances_over_the_sites_or_the_mask(H, W):
    fg = np.ones((H, W), np.uint8)
    fg[H // 2, W // 3] = 0
    yy, xx = np.mgrid[0:H, 0:W]
    want = (yy - H // 2) ** 2 + (xx - W // 3) ** 2   # one site: exact
    T = iwpp.DistanceTransform(H, W)
    out = torch.empty((H, W), dtype=torch.int32, device="cuda")
    assert T(torch.from_numpy(fg).cuda(), out, out, 8) == 0 and T.status() == 0
    assert np.array_equal(out.cpu().numpy(), want)
    mask = out.view(torch.uint8).reshape(-1)[:H * W].view(H, W)   # the mask where the distances go
    mask.copy_(torch.from_numpy(fg))
    site = torch.empty_like(out)
    assert T(mask, site, out, 8) == 0 and T.status() == 0
    assert np.array_equal(out.cpu().numpy(), want)
    assert np.all(site.cpu().numpy() == ((H // 2) << 16 | (W // 3)))

"""GPU: the scan kernel at the edges of its strips and spans: widths around multiples of the 8-pixel
span (aligned spans, words joined by shifts, pixel by pixel), heights around its 16-row strips.
One pixel that can rise must queue its tile (the result then equals the oracle's), one pixel
above the mask must be reported."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle
from paper_1605_00930_gb300 import iwpp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [np.uint8, np.uint16])
@pytest.mark.parametrize("W", [1, 3, 7, 8, 9, 63, 64, 66, 71, 72, 129, 131])
def test_scan_edges(dtype, W):
    rng = np.random.default_rng(W)
    mv = int(np.iinfo(dtype).max)
    for H in (1, 2, 15, 16, 17, 65):
        spots = {(0, 0), (H - 1, W - 1), (0, W - 1), (H - 1, 0), (H // 2, W // 2)}
        for conn, op in ((8, "dilate"), (4, "erode")):
            R = iwpp.Reconstructor(H, W, torch.uint8 if dtype == np.uint8 else torch.uint16)
            flat = np.full((H, W), mv // 2, dtype)
            for y, x in spots:   # one pixel of a flat image below (dilate) / above (erode) its mask
                mk = flat.copy()
                mk[y, x] = mv // 2 - 9 if op == "dilate" else mv // 2 + 9
                m, I = torch.from_numpy(mk.copy()).cuda(), torch.from_numpy(flat).cuda()
                assert R(m, I, conn, op) == 0 and R.status() == 0
                assert np.array_equal(m.cpu().numpy(), oracle.reconstruct(mk, flat, conn, op)), (H, y, x, op)
                mk[y, x] = mv // 2 + 9 if op == "dilate" else mv // 2 - 9   # on the wrong side of it
                assert R(torch.from_numpy(mk).cuda(), I, conn, op) == 0 and R.status() == 2, (H, y, x, op)
            mask = rng.integers(0, mv + 1, (H, W)).astype(dtype)
            mk = np.where(rng.random((H, W)) < 0.9, mask, 0 if op == "dilate" else mv).astype(dtype)
            m = torch.from_numpy(mk).cuda()
            assert R(m, torch.from_numpy(mask).cuda(), conn, op) == 0 and R.status() == 0
            assert np.array_equal(m.cpu().numpy(), oracle.reconstruct(mk, mask, conn, op)), (H, op)

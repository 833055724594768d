"""GPU: the persistent kernel's build for single dilations of many tiles (at least 8192): images
that are long rather than large, both sides of the limit, both pixel types and connectivities, and
three rows of tiles, so that tiles have all eight neighbours."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle
from paper_1605_00930_gb300 import iwpp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 64 * 8191), (1, 64 * 8191 + 1), (66, 64 * 4095 + 3), (64 * 8192 + 5, 2)])
@pytest.mark.parametrize("dtype,conn", [(np.uint8, 8), (np.uint16, 8), (np.uint8, 4), (np.uint16, 4)])
def test_long_images(shape, dtype, conn):
    check(shape, dtype, conn)


@pytest.mark.parametrize("dtype,conn", [(np.uint8, 8), (np.uint16, 4)])
def test_three_rows_of_tiles(dtype, conn):
    check((150, 64 * 2760 + 9), dtype, conn)


def check(shape, dtype, conn):
    rng = np.random.default_rng([shape[0], shape[1], conn])
    mv = int(np.iinfo(dtype).max)
    mask = rng.integers(mv // 4, mv + 1, shape).astype(dtype)
    mask[rng.random(shape) < 0.02] = 0
    marker = np.where(rng.random(shape) < 0.002, mask, 0).astype(dtype)
    R = iwpp.Reconstructor(*shape, torch.uint8 if dtype == np.uint8 else torch.uint16)
    m = torch.from_numpy(marker).cuda()
    assert R(m, torch.from_numpy(mask).cuda(), conn, "dilate") == 0 and R.status() == 0
    assert np.array_equal(m.cpu().numpy(), oracle.reconstruct(marker, mask, conn, "dilate"))

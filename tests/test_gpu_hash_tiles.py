"""GPU parity of the window hashes at the edges of both tile sizes: windows of up
to 256 bytes are hashed in tiles of 2048 bytes, longer ones in tiles of 8192."""

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

from gpu_util import require_gpu, to_device  # noqa: E402
from paper_1810_01051_gb300 import rk  # noqa: E402

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("L", [1, 2, 15, 16, 17, 31, 32, 33, 128, 255, 256, 257, 258, 512, 4096])
@pytest.mark.parametrize("base_log2", [8, 13])
def test_tile_edges(L, base_log2):
    tile = 2048 if L <= 256 else 8192
    per = (tile - L + 1) // 32 * 32  # windows of a tile
    rng = np.random.default_rng(L + base_log2)
    for tiles in (1, 2, 5):
        for off in (-1, 0, 1, 31):
            windows = tiles * per + off
            n = windows + L - 1
            text = rng.integers(0, 256, n, dtype=np.uint8)
            text[rng.random(n) < 0.3] = 255
            d = to_device(text, (7 * tiles + off) % 16)
            out = torch.full((windows + 1,), -1, dtype=torch.int64, device="cuda")
            rk.rk_window_hashes_device(d, n, L, base_log2, out)
            got = out.cpu().numpy()
            assert np.array_equal(got[:-1].view(np.uint64),
                                  oracle.window_hashes(text, L, 1 << base_log2)), (L, tiles, off)
            assert got[-1] == -1  # one past the last window is not written

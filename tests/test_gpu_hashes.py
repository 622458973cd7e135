"""GPU parity of the window hashes where the tiled prefix kernel can go wrong:
window lengths at the edges of a thread's 16 bytes, a warp's 512 and the
longest allowed, texts that end at a tile's edge or one byte off it, every
kind of text alignment, and the bases with a rotation of their own."""

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


TILE = 8192


@pytest.mark.parametrize("L", [1, 2, 15, 16, 17, 511, 512, 513, 4095, 4096])
@pytest.mark.parametrize("base_log2", [8, 1, 60])
def test_tile_edges(L, base_log2):
    rng = np.random.default_rng(L * 61 + base_log2)
    per = (TILE - L + 1) // 32 * 32  # windows of a tile
    for i, n in enumerate((L, L + 1, per + L - 2, per + L - 1, per + L, 2 * per + L + 5)):
        text = rng.integers(0, 256, n, dtype=np.uint8)
        text[rng.random(n) < 0.3] = 255
        expect = oracle.window_hashes(text, L, 1 << base_log2)
        d = to_device(text, (5 * i + L) % 16)
        out = torch.full((n - L + 2,), -1, dtype=torch.int64, device="cuda")
        rk.rk_window_hashes_device(d, n, L, base_log2, out)
        got = out.cpu().numpy()
        assert np.array_equal(got[:-1].view(np.uint64), expect), (L, n)
        assert got[-1] == -1  # one past the last window is not written

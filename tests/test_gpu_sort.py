"""GPU parity of the single-launch sort on key lists made here (rk_sort_device
reads only the count and the keys): even and skewed spreads over the cells,
lists crowded into few cells (sorted by the radix passes instead), sizes at
the edges of a tile and of the one-CTA sort, texts and pattern counts that
leave one field empty.  Expected order: numpy's sort."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from gpu_util import require_gpu  # noqa: E402
from paper_1810_01051_gb300 import rk  # noqa: E402

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def keys_of(ids, xs):
    return (ids.astype(np.uint64) << np.uint64(40)) | xs.astype(np.uint64)


def make(spread, m, n, k, rng):
    """About m distinct keys with ids below k and offsets below n, shuffled."""
    ids = rng.integers(0, k, m)
    if spread == "even":
        xs = rng.integers(0, n, m)
    elif spread == "one_id":  # nine in ten matches are of one pattern
        ids = np.where(rng.random(m) < 0.9, k - 1, ids)
        xs = rng.integers(0, n, m)
    elif spread == "crowded":  # all matches in one stretch of the text
        xs = n - 1 - rng.integers(0, min(n, 4 * m // k + 64), m)
    else:  # a few in each cell of one corner, as from a text of one letter
        xs = rng.integers(0, max(1, n // 64), m)
    keys = np.unique(keys_of(ids, xs))
    return rng.permutation(keys)


@pytest.mark.parametrize("spread", ["even", "one_id", "crowded", "corner"])
@pytest.mark.parametrize("m,n,k", [
    (2, 10, 3), (37, 100, 1), (2048, 1 << 20, 7), (2049, 1 << 20, 7), (2050, (1 << 30) + 1, 100),
    (5000, 5000, 1), (70000, (1 << 32) + 5, 10000), (1 << 17, 1 << 24, 3),
    (700_001, (1 << 30) - 3, 100), (3_000_000, (1 << 39) + 1, 1000),
])
def test_sort_spreads(spread, m, n, k):
    rng = np.random.default_rng(m + n + len(spread))
    keys = make(spread, m, n, k, rng)
    table = rk.rk_build([b"%06d" % i for i in range(k)])
    try:
        for cap in (keys.size, keys.size + 3000):
            d = torch.zeros(cap, dtype=torch.int64, device="cuda")
            d[:keys.size] = torch.from_numpy(keys.view(np.int64)).cuda()
            info = torch.tensor([keys.size, 0], dtype=torch.int64, device="cuda")
            wsb = rk.rk_workspace_bytes(table, cap)
            ws = torch.full((max(wsb, 16),), 0xA5, dtype=torch.uint8, device="cuda")
            rk.rk_sort_device(table, n, d, cap, info, ws, wsb)
            torch.cuda.synchronize()
            got = d.cpu().numpy().view(np.uint64)
            assert int(info[1]) == rk.RK_OK
            assert np.array_equal(got[:keys.size], np.sort(keys)), (spread, cap)
            assert not got[keys.size:].any()  # nothing past the list is touched
    finally:
        rk.rk_destroy(table)


@pytest.mark.parametrize("spread", ["even", "one_id"])
@pytest.mark.parametrize("m", [511 * 8, 4096, 4097, (1 << 18) - 1, 1 << 18, (1 << 18) + 1])
@pytest.mark.parametrize("spare", [0, 1, 400_000])
def test_sort_cell_counts(spread, m, spare):
    """Sizes where the number of CTAs and of cells per key change; the cells also
    depend on the workspace, so on the room beyond the list."""
    n, k = 1 << 30, 100
    rng = np.random.default_rng(m + spare)
    keys = make(spread, m + m // 8, n, k, rng)[:m]
    table = rk.rk_build([b"%06d" % i for i in range(k)])
    try:
        cap = keys.size + spare
        d = torch.zeros(cap, dtype=torch.int64, device="cuda")
        d[:keys.size] = torch.from_numpy(keys.view(np.int64)).cuda()
        info = torch.tensor([keys.size, 0], dtype=torch.int64, device="cuda")
        wsb = rk.rk_workspace_bytes(table, cap)
        ws = torch.full((wsb + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
        rk.rk_sort_device(table, n, d, cap, info, ws, wsb)
        torch.cuda.synchronize()
        got = d.cpu().numpy().view(np.uint64)
        assert int(info[1]) == rk.RK_OK
        assert np.array_equal(got[:keys.size], np.sort(keys))
        assert not got[keys.size:].any()
        assert bool((ws[wsb:] == 0xA5).all())  # nothing past the workspace
    finally:
        rk.rk_destroy(table)

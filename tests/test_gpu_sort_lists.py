"""GPU parity of rk_sort_device on key lists that no one search gives: keys
outside the fields that the text length and the pattern count allow, and keys
that occur more than once; and lists whose keys lie close together, which are
sorted by the radix passes."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from gpu_util import require_gpu  # noqa: E402
from paper_1810_01051_gb300 import rk  # noqa: E402

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def sort_keys(keys, n, k, spare=0):
    """keys sorted by rk_sort_device for a text of n bytes and k patterns; the
    workspace and what lies after it are checked to be kept apart."""
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
        assert int(info[1]) == rk.RK_OK and int(info[0]) == keys.size
        assert bool((ws[wsb:] == 0xA5).all())
        got = d.cpu().numpy().view(np.uint64)
        assert not got[keys.size:].any()
        return got[:keys.size]
    finally:
        rk.rk_destroy(table)


def field_order(keys, n, k):
    """A stable sort by the bytes that the offsets below n and the ids below k
    occupy: the order of any key list, ascending where those bytes hold the
    whole key."""
    lo = -(-int(n - 1).bit_length() // 8) * 8
    hi = -(-int(k - 1).bit_length() // 8) * 8
    mask = np.uint64((((1 << hi) - 1) << 40) | ((1 << lo) - 1))
    return keys[np.argsort(keys & mask, kind="stable")]


@pytest.mark.parametrize("bad", ["id", "id of all ones", "offset", "one key of all ones"])
@pytest.mark.parametrize("m,n,k", [(2, 100, 3), (700, 1 << 20, 7), (2048, 1 << 20, 1),
                                   (2049, 1 << 20, 7), (70_001, (1 << 30) - 3, 100),
                                   (700_001, 1 << 24, 3)])
def test_keys_outside_the_fields(m, n, k, bad):
    rng = np.random.default_rng(m + len(bad))
    ids = rng.integers(0, k, m).astype(np.uint64)
    xs = rng.integers(0, n, m).astype(np.uint64)
    some = rng.random(m) < 0.3
    if bad == "id":
        ids[some] += np.uint64(k)
    elif bad == "id of all ones":
        ids[some] = np.uint64((1 << 24) - 1)
    elif bad == "offset":
        xs[some] = rng.integers(0, 1 << 40, int(some.sum())).astype(np.uint64)
    else:
        ids[m // 2], xs[m // 2] = np.uint64((1 << 24) - 1), np.uint64((1 << 40) - 1)
    keys = (ids << np.uint64(40)) | xs
    for spare in (0, 3000):
        got = sort_keys(keys, n, k, spare)
        assert np.array_equal(got, field_order(keys, n, k)), (spare, bad)


@pytest.mark.parametrize("copies", [2, 3, 40])
@pytest.mark.parametrize("m", [2, 3, 64, 2047, 2048, 2049, 4097, 70_001, (1 << 18) + 5])
def test_equal_keys(m, copies):
    """Every copy of a key stays in the list, the field's largest and smallest
    keys among them."""
    n, k = 1 << 26, 8
    rng = np.random.default_rng(m + copies)
    own = rng.integers(0, n, -(-m // copies)).astype(np.uint64)
    own |= rng.integers(0, k, own.size).astype(np.uint64) << np.uint64(40)
    own[0] = (np.uint64(k - 1) << np.uint64(40)) | np.uint64(n - 1)
    own[-1] = 0 if own.size > 1 else own[-1]
    keys = rng.permutation(np.repeat(own, copies)[:m])
    for spare in (0, 3000):
        assert np.array_equal(sort_keys(keys, n, k, spare), np.sort(keys)), spare


def clumped(m, n, k, per_cell, rng):
    """About m distinct keys with about per_cell to each 2^15 offsets of an id."""
    span = int(min(n, max(64, m * 2**15 // (k * per_cell))))
    keys = rng.integers(0, k, m).astype(np.uint64) << np.uint64(40)
    keys |= (rng.integers(0, span, m) + (n - span) // 2).astype(np.uint64)
    return rng.permutation(np.unique(keys))


@pytest.mark.parametrize("per_cell", [8, 90, 110, 130, 500, 5000])
@pytest.mark.parametrize("m", [2049, 5000, 300_001, 5_000_000])
def test_clumped_keys(m, per_cell):
    """On both sides of the mean cell size above which the radix passes run."""
    n, k = 1 << 30, 100
    keys = clumped(m, n, k, per_cell, np.random.default_rng(m + per_cell))
    assert np.array_equal(sort_keys(keys, n, k, 1000), np.sort(keys))


def test_clumped_keys_take_no_longer_than_the_passes():
    """A few hundred keys to a cell: the radix passes take about twice as long as
    cells do for evenly spread keys; comparing within the cells, six times."""
    n, k, m = 1 << 30, 100, 5_000_000
    rng = np.random.default_rng(3)
    table = rk.rk_build([b"%06d" % i for i in range(k)])
    try:
        wsb = rk.rk_workspace_bytes(table, m)  # m: the most there are
        ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
        took = []
        for keys in (clumped(m, n, k, 1, rng), clumped(m, n, k, 700, rng)):
            src = torch.from_numpy(keys.view(np.int64)).cuda()
            d = torch.empty_like(src)
            info = torch.tensor([src.numel(), 0], dtype=torch.int64, device="cuda")
            best = 1e9
            for _ in range(8):
                d.copy_(src)
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                a.record()
                rk.rk_sort_device(table, n, d, src.numel(), info, ws, wsb)
                b.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b))
            took.append(best)
        assert took[1] < 4 * took[0], took
    finally:
        rk.rk_destroy(table)

"""GPU parity of scans that list their candidates (rk_scan_device_ws, whatever
route a search of the same text would take) against the oracle, with what the
list may hold: only windows that start with the prefix of some pattern."""

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

from gpu_util import (assert_same, gpu_search, keys_to_pairs, require_gpu,  # noqa: E402
                      to_device)
from paper_1810_01051_gb300 import rk  # noqa: E402

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def listed_scan(patterns, text, misalign=0, cap=1 << 18, **opts):
    """Sorted (ids, offsets) and the number of candidates listed."""
    n = int(text.size)
    table = rk.rk_build(list(patterns), **opts)
    try:
        d = to_device(text, misalign)
        keys = torch.empty(cap, dtype=torch.int64, device="cuda")
        info = torch.full((2,), -1, dtype=torch.int64, device="cuda")
        sort_b, scan_b = rk.rk_workspace_bytes(table, cap), rk.rk_scan_workspace_bytes(table, n)
        ws = torch.empty(sort_b, dtype=torch.uint8, device="cuda")
        lst = torch.full((scan_b,), 0xFF, dtype=torch.uint8, device="cuda")
        assert rk.rk_scan_launches(table, n, scan_b) == 2
        rk.rk_scan_device_ws(table, d, n, keys, cap, info, lst, scan_b)
        rk.rk_sort_device(table, n, keys, cap, info, ws, sort_b)
        torch.cuda.synchronize()
        count, status = (int(v) for v in info.cpu().tolist())
        assert status == rk.RK_OK and count <= cap
        return keys_to_pairs(keys[:count]), int(lst[:8].view(torch.int64)[0])
    finally:
        rk.rk_destroy(table)


@pytest.mark.parametrize("run", [b"\0" * 8, b"abab" * 3])
@pytest.mark.parametrize("many", [0, 2000])
def test_listed_windows_start_with_a_prefix(run, many):
    """A gram that fills the text and that one pattern has, at one offset behind
    other bytes: the windows it points at start with another prefix."""
    rng = np.random.default_rng(len(run) + many)
    text = np.frombuffer(run * (300_000 // len(run)), np.uint8).copy()
    noise = rng.integers(0, text.size - 64, 2000)
    text[noise] = rng.integers(0, 256, noise.size)
    pats = [b"xyz" + run[:5] + b"\1tail", b"QRSTUVWXYZ"]
    pats += [rng.integers(1, 256, int(L), dtype=np.uint8).tobytes()
             for L in rng.integers(8, 40, many)]
    for i, at in enumerate(rng.integers(0, text.size - 64, 200)):
        p = pats[i % len(pats)]
        text[at:at + len(p)] = np.frombuffer(p, np.uint8)
    expect = oracle.rabin_karp(text, pats)
    words = np.lib.stride_tricks.sliding_window_view(text, 4)
    starts = {p[:4] for p in pats}
    with_prefix = sum(int((words == np.frombuffer(s, np.uint8)).all(1).sum()) for s in
                      starts if s[0] in text)
    for mis in (0, 3):
        got, listed = listed_scan(pats, text, mis, role_step=1)
        assert_same(got, expect, f"mis {mis}")
        assert expect[0].size <= listed <= with_prefix


@pytest.mark.parametrize("opts,lmin,lmax,counts", [
    (dict(), 8, 64, (120, 250, 290, 310, 330)),
    (dict(role_step=1), 8, 64, (80, 200, 300, 336)),
    (dict(role_step=1, sample=1), 8, 40, (300, 420)),
    (dict(role_step=1), 3, 12, (300, 500)),
    (dict(filter=rk.RK_FILTER_NONE), 4, 32, (40, 520)),
])
def test_every_density_of_the_prefix_map(opts, lmin, lmax, counts):
    """Sets whose map is sparse, denser or as dense as it gets, so that their
    tables still fit shared memory: searched in the scan and through the list."""
    rng = np.random.default_rng(lmin + lmax)
    n = 60_000 if "filter" in opts else 300_000
    text = rng.choice(np.frombuffer(b"etaoinsh rdlcum", np.uint8), n)
    for k in counts:
        at = rng.integers(0, n - lmax, k)
        pats = [text[a:a + int(L)].tobytes() for a, L in zip(at, rng.integers(lmin, lmax + 1, k))]
        expect = oracle.rabin_karp(text, pats)
        if "filter" not in opts:
            got, listed = listed_scan(pats, text, 5, **opts)
            assert_same(got, expect, f"listed, {k}")
            assert listed > 0
        assert_same(gpu_search(pats, text, 5, **opts), expect, f"in the scan, {k}")

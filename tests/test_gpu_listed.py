"""GPU parity of scans that list their candidates (rk_scan_device_ws, whatever
route a search of the same text would take) against the oracle, with what the
list may hold: only windows that start with the prefix of some pattern."""

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

import test_gpu_deferred as deferred  # noqa: E402
import test_gpu_roles as roles  # noqa: E402
import test_gpu_sampled as sampled  # noqa: E402
from gpu_util import (assert_same, gpu_search, keys_to_pairs, require_gpu,  # noqa: E402
                      to_device)
from paper_1810_01051_gb300 import rk  # noqa: E402

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def listed_scan(patterns, text, misalign=0, **opts):
    """Sorted (ids, offsets) and the number of candidates listed (None for a table
    that lists none)."""
    n = int(text.size)
    table = rk.rk_build(list(patterns), **opts)
    cap = max(1024, n // 8)
    try:
        d = to_device(text, misalign)
        while True:
            keys = torch.empty(cap, dtype=torch.int64, device="cuda")
            info = torch.full((2,), -1, dtype=torch.int64, device="cuda")
            sort_b, scan_b = rk.rk_workspace_bytes(table, cap), rk.rk_scan_workspace_bytes(table, n)
            ws = torch.empty(sort_b, dtype=torch.uint8, device="cuda")
            lst = torch.full((scan_b,), 0xFF, dtype=torch.uint8, device="cuda")
            lists = rk.rk_scan_launches(table, n, scan_b) == 2
            rk.rk_scan_device_ws(table, d if n else 0, n, keys, cap, info, lst, scan_b)
            rk.rk_sort_device(table, n, keys, cap, info, ws, sort_b)
            torch.cuda.synchronize()
            count, status = (int(v) for v in info.cpu().tolist())
            assert status == rk.RK_OK, rk.strerror(status)
            if count <= cap:
                break
            cap = count
        listed = int(lst[:8].view(torch.int64)[0]) if lists else None
        assert lists == (n > 0 and opts.get("filter") != rk.RK_FILTER_NONE)
        return keys_to_pairs(keys[:count]), listed
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


@pytest.mark.parametrize("alphabet,k,lmin,lmax", [
    (b"ABCDEFGHIJKLMNOPQRST", 40, 1, 3), (b"ACGT", 40, 2, 6), (b"ACGT", 40, 1, 1),
    (b"etaoinshr ", 200, 2, 4), (b"ACGT", 8, 1, 2), (b"ACGT", 60, 3, 8), (b"ACGT", 60, 3, 9),
])
def test_short_patterns_of_shared_prefixes(alphabet, k, lmin, lmax):
    """Many patterns of one prefix and length, repeated ones among them, beside
    prefixes with one."""
    rng = np.random.default_rng(k + lmax)
    sym = np.frombuffer(alphabet, np.uint8)
    text = rng.choice(sym, 50_003)
    pats = [rng.choice(sym, int(L)).tobytes() for L in rng.integers(lmin, lmax + 1, k)]
    pats.append(pats[0])
    expect = oracle.rabin_karp(text, pats)
    for opts in (dict(), dict(base_log2=1), dict(tile_bytes=1024, stages=2, warps=2)):
        got, listed = listed_scan(pats, text, 5, **opts)
        assert_same(got, expect, f"listed {opts}")
        assert listed > 0
        assert_same(gpu_search(pats, text, 5, **opts), expect, f"in the scan {opts}")


# ---- the tests of the deferred, sampled and role-filter scans, always listed ----

@pytest.fixture
def listing(monkeypatch):
    """deferred_search of those tests by rk_scan_device_ws, with a list that is
    used: at least one candidate wherever something matches."""
    def search(patterns, text, misalign=0, via_search=True, **opts):
        got, listed = listed_scan(patterns, text, misalign, **opts)
        assert listed is None or listed >= min(1, got[0].size)
        return got
    for module in (deferred, sampled, roles):
        monkeypatch.setattr(module, "deferred_search", search)


@pytest.mark.parametrize("seed", range(18))
def test_fuzz_sampled(listing, seed):
    sampled.test_fuzz_sampled(seed)


@pytest.mark.parametrize("seed", range(24))
def test_fuzz_roles(listing, seed):
    roles.test_fuzz_roles(seed)


@pytest.mark.parametrize("tail", range(0, 17))
def test_text_ends(listing, tail):
    sampled.test_text_end_offsets(tail)
    roles.test_text_end_offsets(tail)
    if tail:
        deferred.test_text_end_reads(tail)


def test_edges(listing):
    sampled.test_repeated_grams_and_shortest_patterns()
    roles.test_four_byte_patterns_at_every_offset()
    roles.test_forced_step(2)
    roles.test_forced_step(4)


def test_full_lists(listing):
    sampled.test_list_overflow_sampled()
    deferred.test_list_overflow_verified_in_scan()
    roles.test_every_window_a_candidate()


@pytest.mark.parametrize("tail", range(0, 17))
def test_long_windows_at_the_text_end(tail):
    """The verification kernel reads a window 32 bytes at a time after its first 8:
    lengths around those steps, ending with the text and before it."""
    rng = np.random.default_rng(700 + tail)
    n = 6000 + tail
    text = rng.integers(0, 3, n, dtype=np.uint8) + ord("a")
    lens = (7, 8, 9, 15, 16, 17, 39, 40, 41, 71, 72, 73, 103, 104, 105, 300)
    pats = [text[n - L:].tobytes() for L in lens] + [text[s:s + L].tobytes() for s, L in
                                                     enumerate(lens)]
    # one wrong byte, in every place of the last step
    pats += [text[n - 73:n - 73 + j].tobytes() + b"z" + text[n - 72 + j:].tobytes()
             for j in (7, 8, 39, 40, 41, 70, 71, 72)]
    expect = oracle.bruteforce(text, pats)
    for mis in range(0, 16, 3):
        for opts in (dict(), dict(role_step=1)):
            got, listed = listed_scan(pats, text, mis, **opts)
            assert_same(got, expect, f"mis {mis} {opts}")
            assert listed > 0

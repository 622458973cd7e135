"""Which route a search given room for a list takes: the list's count is
written when it lists and left alone when its scan completes the survivors.
Either way the matches are the oracle's."""

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

from gpu_util import assert_same, keys_to_pairs, require_gpu, to_device  # noqa: E402
from paper_1810_01051_gb300 import rk  # noqa: E402

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


MIB = 1 << 20
WORDS = b"etaoinshrdlcumwfgypbvkjxqz "


def random_text(alphabet, n, seed):
    return np.random.default_rng(seed).choice(np.frombuffer(alphabet, np.uint8), n)


def random_patterns(alphabet, k, lmin, lmax, seed):
    rng = np.random.default_rng(seed)
    sym = np.frombuffer(alphabet, np.uint8)
    return [rng.choice(sym, int(L)).tobytes() for L in rng.integers(lmin, lmax + 1, k)]


def search(table, text, cap=1 << 18):
    """The sorted matches, and whether the list was used."""
    n = int(text.size)
    d = to_device(text, 3)
    keys = torch.empty(cap, dtype=torch.int64, device="cuda")
    info = torch.full((2,), -1, dtype=torch.int64, device="cuda")
    sort_b, scan_b = rk.rk_workspace_bytes(table, cap), rk.rk_scan_workspace_bytes(table, n)
    ws = torch.full((sort_b + scan_b,), 0xA5, dtype=torch.uint8, device="cuda")
    rk.rk_search_device(table, d, n, keys, cap, info, ws, sort_b + scan_b)
    torch.cuda.synchronize()
    count, status = (int(v) for v in info.cpu().tolist())
    assert status == rk.RK_OK and count <= cap
    listed = not bool((ws[sort_b:sort_b + 8] == 0xA5).all())
    return keys_to_pairs(keys[:count]), listed


CASES = [
    # alphabet, patterns, lengths, options, text bytes, whether listed
    ("few probes", b"ACGT", 8, (16, 16), {}, MIB, False),
    ("many probes", b"ACGT", 128, (16, 16), {}, MIB, True),
    ("many probes, short text", b"ACGT", 256, (16, 16), {}, 64 << 10, True),
    ("some probes, short text", b"ACGT", 32, (16, 16), {}, MIB, False),
    ("some probes, longer text", b"ACGT", 32, (16, 16), {}, 8 * MIB, True),
    ("words", WORDS, 100, (4, 32), {}, MIB, False),
    ("words, long text", WORDS, 100, (7, 32), {}, 48 * MIB + 1, True),
    ("three letters on", WORDS, 100, (3, 12), {}, MIB, False),
    ("every position", b"ACGT", 100, (16, 16), dict(role_step=1, sample=1), MIB, False),
    ("sampled", WORDS, 5000, (16, 40), dict(role_step=1), 4 * MIB, False),
    ("sampled, longer text", WORDS, 5000, (16, 40), dict(role_step=1), 4 * MIB + 1, True),
    ("tables in L2", WORDS, 1500, (7, 32), {}, MIB, True),
    ("no filter", WORDS, 20, (4, 12), dict(filter=rk.RK_FILTER_NONE), 64 << 10, False),
]


@pytest.mark.parametrize("name,alphabet,k,lens,opts,n,lists", CASES, ids=[c[0] for c in CASES])
def test_route(name, alphabet, k, lens, opts, n, lists):
    text = random_text(alphabet, n, k)
    pats = random_patterns(alphabet, k, *lens, seed=k + n)
    rng = np.random.default_rng(n)
    for i, at in enumerate(rng.integers(0, n - 64, 500)):
        p = pats[i % k]
        text[at:at + len(p)] = np.frombuffer(p, np.uint8)
    table = rk.rk_build(pats, **opts)
    try:
        got, listed = search(table, text)
        assert listed == lists
        # (the oracle on a part of the longer texts)
        m = min(n, 2 * MIB)
        ids, offs = oracle.rabin_karp(text[:m], pats)
        lens_of = np.array([len(p) for p in pats])
        inside = got[1].astype(np.int64) + lens_of[got[0]] <= m
        assert_same((got[0][inside], got[1][inside]), (ids, offs), name)
    finally:
        rk.rk_destroy(table)

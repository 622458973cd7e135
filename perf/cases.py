"""The work a user of this library has it do, as cases that can be timed.

A case names what is searched (``kind``), through which entry point (``api``)
and at which sizes.  ``listed()`` gives the fixed cases, ``draw(rng)`` more of
the same ranges, ``prepare(case, seed)`` what a program holds before the call
(text, table, output and workspace), ``run(state)`` one call and its outputs,
``work(case)`` the bytes that call cannot do without.

Texts are drawn on the GPU from the seed.  Plants never overlap (each has its
own stretch of the text), so that a seed gives the same bytes every time.  All
outputs are whole numbers (match keys, counts, hashes): they are compared for
equality, so no 64-bit reference values are given here.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_1810_01051_gb300 import rk
from paper_1810_01051_gb300.matcher import Matcher

MIB = 1 << 20

#: letters by falling frequency, weight 1/rank, and a space every six characters
LETTERS = b"etaoinshrdlcumwfgypbvkjxqz"
LETTER_W = np.array([1.0 / r for r in range(1, 27)])
LETTER_P = np.append(LETTER_W / LETTER_W.sum() * (5.0 / 6.0), 1.0 / 6.0)

ALPHABETS = {
    "dna": (np.frombuffer(b"ACGT", np.uint8), np.full(4, 0.25)),
    "words": (np.frombuffer(LETTERS + b" ", np.uint8), LETTER_P),
    "bytes": (np.arange(256, dtype=np.uint8), np.full(256, 1.0 / 256)),
    "letters": (np.frombuffer(b"ABCDEFGHIJKLMNOPQRST", np.uint8), np.full(20, 0.05)),
}


def listed():
    return [
        # One search of a short DNA text for a few probes, buffers kept by the
        # caller: the latency of scan, verification and sort.
        dict(name="dna_1MiB_8x16", api="search", kind="dna", n=MIB, k=8, lmin=16, lmax=16,
             plants=50, mis=0),
        # The convenience class on a text of a few pages, as a Python program
        # calls it (output and workspace allocated inside): the smallest call.
        dict(name="matcher_words_40kB", api="matcher", kind="words", n=40_003, k=100, lmin=4,
             lmax=32, plants=1, mis=0),
        # The large plain scan: English-like text, 100 patterns of 4..32 letters.
        dict(name="words_1GiB_100x4-32", api="search", kind="words", n=1 << 30, k=100, lmin=4,
             lmax=32, plants=1074, mis=0),
        # Keywords from three letters on: prefixes shorter than four bytes and
        # many matches, an odd length and an unaligned text.
        dict(name="words_64MB_100x3-12", api="search", kind="words", n=64_000_001, k=100, lmin=3,
             lmax=12, plants=64, mis=3),
        # The signature set: 10,000 byte signatures over 4 GiB of binary data.
        dict(name="bytes_4GiB_10000x8-64", api="search", kind="bytes", n=4 << 30, k=10000, lmin=8,
             lmax=64, plants=1000, mis=0),
        # A smaller signature set over a file image, the result as match records.
        dict(name="records_bytes_256MiB_1000x8-64", api="records", kind="bytes", n=256 * MIB,
             k=1000, lmin=8, lmax=64, plants=64, mis=0),
        # Long DNA probes (the paper's lengths, 25..800 bytes) in one text.
        dict(name="dna_64MB_16x25-800", api="search", kind="dna", n=64_000_000, k=16, lmin=25,
             lmax=800, plants=100, mis=0),
        # The search that allocates nothing (single-kernel scan, fixed scratch),
        # at an odd length from an unaligned address.
        dict(name="noalloc_words_33MB_100x4-32", api="noalloc", kind="words", n=33_000_017, k=100,
             lmin=4, lmax=32, plants=33, mis=5),
        # A host text searched end to end: copy in, scan, sort, copy out.
        dict(name="host_words_256MiB_100x4-32", api="host", kind="words", n=256 * MIB, k=100,
             lmin=4, lmax=32, plants=268, mis=0),
        # A thousand texts of 1 KiB..16 MiB, each with a pattern set of its own,
        # in one graph launch.
        dict(name="batch_1024x1KiB-16MiB", api="batch", kind="letters", items=1024, min_len=1024,
             max_len=16 * MIB, k_max=256, lmin=4, lmax=48),
        # Many small requests at once (messages, records): launch and per-text
        # costs rather than bytes.
        dict(name="batch_4096x1-64KiB", api="batch", kind="letters", items=4096, min_len=1000,
             max_len=64 << 10, k_max=64, lmin=4, lmax=48),
        # The Rabin hash of every window of a text.
        dict(name="hashes_128MiB_L16", api="hashes", kind="bytes", n=128 * MIB, L=16, base_log2=8,
             mis=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    api = rng.choice(["search", "search", "search", "search", "matcher", "records", "noalloc",
                      "host", "batch", "batch", "hashes"])
    if api == "batch":
        lo = rng.choice([1000, 1024, 4096])
        return dict(api=api, kind=rng.choice(["letters", "bytes"]), items=_log(rng, 32, 1024),
                    min_len=lo, max_len=_log(rng, 32 << 10, 16 * MIB), k_max=_log(rng, 4, 256),
                    lmin=4, lmax=rng.randint(8, 64))
    if api == "hashes":
        return dict(api=api, kind=rng.choice(["bytes", "dna"]), n=_log(rng, 64 << 10, 128 * MIB),
                    L=_log(rng, 1, 400), base_log2=rng.choice([8, 8, 1, 13]),
                    mis=rng.randrange(16))
    kind = rng.choice(["dna", "words", "bytes"])
    # pattern lengths: short keywords and probes, ordinary ones, long ones
    lmin = rng.choice({"dna": [7, 16, 25], "words": [3, 4, 5, 8], "bytes": [4, 6, 8, 16]}[kind])
    lmax = lmin + _log(rng, 1, {"dna": 775, "words": 28, "bytes": 56}[kind]) - 1
    k = _log(rng, 1, {"dna": 64, "words": 200, "bytes": 10000}[kind])
    top = {"search": 1 << 30, "matcher": 64 * MIB, "records": 256 * MIB, "noalloc": 256 * MIB,
           "host": 256 * MIB}[api]
    if lmin < 4:
        top = min(top, 64 * MIB)
    n = max(_log(rng, 4096, top), 4 * lmax)
    k = min(k, n // (lmax + 1))  # a place for every pattern
    c = dict(api=api, kind=kind, n=n, k=k, lmin=lmin, lmax=lmax,
             plants=max(1, min(1000, n // (k * 1000))), mis=rng.randrange(16))
    # the search that allocates nothing holds 2^20 matches
    while api == "noalloc" and 4 * _chance_matches(c) > rk.RK_NOALLOC_MAX_KEYS // 2:
        c["n"] //= 2
    return c


# ------------------------------------------------------------------ sizes

def _plants_per_pattern(c):
    """Plants of each pattern that fit, each in its own stretch of the text."""
    return min(c["plants"], c["n"] // (c["k"] * (c["lmax"] + 1)))


def _chance_matches(c):
    """Matches of unplanted text that chance gives."""
    same = float((ALPHABETS[c["kind"]][1] ** 2).sum())
    lens = range(c["lmin"], c["lmax"] + 1)
    return c["k"] * c["n"] * sum(same ** L for L in lens) / len(lens)


def _capacity(c):
    """Output room a program gives the search: about one match in 128 bytes
    of English-like text (one in eight with patterns below four letters), else
    one in 256, and well above the matches expected."""
    per = 256 if c["kind"] != "words" else 8 if c["lmin"] < 4 else 128
    cap = max(4096, c["n"] // per,
              int(1.5 * c["k"] * _plants_per_pattern(c) + 4 * _chance_matches(c)))
    return min(cap, rk.RK_NOALLOC_MAX_KEYS) if c["api"] == "noalloc" else cap


def _item_lens(c):
    """Log-uniform text lengths: the middles of equal shares of the range."""
    u = (np.arange(c["items"]) + 0.5) / c["items"]
    return np.exp(math.log(c["min_len"])
                  + u * (math.log(c["max_len"]) - math.log(c["min_len"]))).astype(np.int64)


def work(case):
    c = case
    if c["api"] == "hashes":
        return dict(bytes=c["n"] + 8 * (c["n"] - c["L"] + 1), flops=0)
    if c["api"] == "batch":
        total = int(_item_lens(c).sum())
        # each of (1 + k_max) / 2 patterns is planted once in 10^5 bytes
        return dict(bytes=total + int(8 * total * 1e-5 * (1 + c["k_max"]) / 2), flops=0)
    key = 16 if c["api"] == "records" else 8
    found = c["k"] * _plants_per_pattern(c) + _chance_matches(c)
    return dict(bytes=c["n"] + int(key * found), flops=0)


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _text(kind, n, g, out=None):
    """n characters of the alphabet, with its frequencies, on the GPU."""
    out = torch.empty(n, dtype=torch.uint8, device="cuda") if out is None else out
    if kind == "bytes":
        return out.random_(0, 256, generator=g)
    sym, p = ALPHABETS[kind]
    at = np.searchsorted(np.cumsum(p), (np.arange(65536) + 0.5) / 65536, side="right")
    lut = torch.from_numpy(sym[np.minimum(at, sym.size - 1)].copy()).cuda()
    for s in range(0, n, 64 * MIB):
        e = min(n, s + 64 * MIB)
        u = torch.randint(0, 65536, (e - s,), dtype=torch.int32, device="cuda", generator=g)
        torch.index_select(lut, 0, u, out=out[s:e])
    return out


def _patterns(kind, k, lmin, lmax, rng):
    """k patterns, lengths uniform in lmin..lmax, as a padded matrix and lengths."""
    sym, p = ALPHABETS[kind]
    at = np.searchsorted(np.cumsum(p), rng.random((k, lmax)), side="right")
    return sym[np.minimum(at, sym.size - 1)], rng.integers(lmin, lmax + 1, k)


def _as_bytes(mat, lens):
    return [row[:L].tobytes() for row, L in zip(mat, lens)]


def _plant(text, pos, ids, mat, lens):
    """Write pattern ids[i] at text[pos[i]...] (GPU tensors; plants are disjoint)."""
    width = mat.shape[1]
    col = torch.arange(width, device="cuda")
    step = max(1, (16 * MIB) // width)
    for s in range(0, pos.numel(), step):
        i = ids[s:s + step]
        keep = col[None, :] < lens[i][:, None]
        text[(pos[s:s + step][:, None] + col[None, :])[keep]] = mat[i][keep]


def _spread(count, n, width, g):
    """count disjoint places of `width` bytes in a text of n bytes."""
    stride = n // count
    jitter = torch.rand(count, generator=g, device="cuda", dtype=torch.float64)
    return torch.arange(count, device="cuda") * stride + (jitter * (stride - width + 1)).long()


class Handle:
    """A library handle, destroyed with its last reference (a handle that it
    uses is kept with it)."""

    def __init__(self, destroy, value, uses=None):
        self.destroy, self.value, self.uses = destroy, value, uses

    def __del__(self):
        self.destroy(self.value)


class State:
    """Buffers and handles of a case."""

    def __init__(self, case):
        self.case = case


class _Device:
    """Device memory owned by a batch engine, for torch.as_tensor (which
    keeps this object, and so the engine, as long as the tensor)."""

    def __init__(self, owner, ptr, n):
        self.owner = owner
        self.__cuda_array_interface__ = dict(data=(ptr, False), shape=(n,), typestr="<i8",
                                             version=2)


def prepare(case, seed):
    s = State(case)
    if case["api"] == "batch":
        _prepare_batch(s, case, seed)
        return s
    g, rng = _gen(seed), np.random.default_rng(seed)
    n, mis = case["n"], case["mis"]
    # the text at `mis` bytes past a 256-byte boundary
    s.text = _text(case["kind"], n, g, torch.empty(n + 64, dtype=torch.uint8,
                                                   device="cuda")[mis:mis + n])
    if case["api"] == "hashes":
        s.out = torch.empty(n - case["L"] + 1, dtype=torch.int64, device="cuda")
        return s
    mat, lens = _patterns(case["kind"], case["k"], case["lmin"], case["lmax"], rng)
    per = _plants_per_pattern(case)
    if per:
        ids = torch.arange(case["k"], device="cuda").repeat(per)
        ids = ids[torch.randperm(ids.numel(), generator=g, device="cuda")]
        _plant(s.text, _spread(ids.numel(), n, case["lmax"], g), ids,
               torch.from_numpy(mat).cuda(), torch.from_numpy(lens).cuda())
    pats = _as_bytes(mat, lens)
    s.cap = _capacity(case)
    if case["api"] == "matcher":
        s.matcher = Matcher(pats)
        s.keys = torch.zeros(s.cap, dtype=torch.int64, device="cuda")
        return s
    s.handle = Handle(rk.rk_destroy, rk.rk_build(pats))
    s.table = s.handle.value
    if case["api"] == "host":
        host = torch.empty(n, dtype=torch.uint8, pin_memory=True)
        host.copy_(s.text)
        s.text = host
        s.keys = torch.zeros(s.cap, dtype=torch.int64, pin_memory=True)
    elif case["api"] == "records":
        s.out = torch.zeros(2 * s.cap, dtype=torch.int64, device="cuda")
    else:
        s.keys = torch.zeros(s.cap, dtype=torch.int64, device="cuda")
        s.info = torch.zeros(2, dtype=torch.int64, device="cuda")
        if case["api"] == "search":
            # room for the sort and for the candidate list, as Matcher gives
            s.ws_bytes = rk.rk_workspace_bytes(s.table, s.cap) + rk.rk_scan_workspace_bytes(
                s.table, n)
            s.ws = torch.empty(s.ws_bytes, dtype=torch.uint8, device="cuda")
    return s


def _prepare_batch(s, c, seed):
    """A batch of texts, each with a pattern set of its own."""
    g, rng = _gen(seed), np.random.default_rng(seed)
    lens = rng.permutation(_item_lens(c))
    # pattern counts spread evenly over 1..k_max
    counts = 1 + rng.permutation(np.arange(c["items"]) * c["k_max"] // c["items"])
    mat, plen = _patterns(c["kind"], int(counts.sum()), c["lmin"], c["lmax"], rng)
    first = np.concatenate([[0], np.cumsum(counts)])
    every = _as_bytes(mat, plen)
    tables = [every[a:b] for a, b in zip(first[:-1], first[1:])]
    # texts in one buffer, each from a 256-byte boundary on
    at = np.concatenate([[0], np.cumsum((lens + 255) // 256 * 256)])
    buf = _text(c["kind"], int(at[-1]) + 64, g)
    pos, ids = [], []
    for i in range(c["items"]):
        # each pattern once in 10^5 bytes (as often as disjoint places allow)
        per = min(int(round(1e-5 * lens[i])), int(lens[i] // (counts[i] * (c["lmax"] + 1))))
        m = per * int(counts[i])
        if m:
            stride = int(lens[i]) // m
            pos.append(at[i] + np.arange(m) * stride
                       + rng.integers(0, stride - c["lmax"] + 1, m))
            ids.append(rng.permutation(np.tile(np.arange(first[i], first[i + 1]), per)))
    if pos:
        _plant(buf, torch.from_numpy(np.concatenate(pos)).cuda(),
               torch.from_numpy(np.concatenate(ids)).cuda(), torch.from_numpy(mat).cuda(),
               torch.from_numpy(plen).cuda())
    total = int(lens.sum())
    cap = 4096 + int(4 * total * 1e-5 * c["k_max"])
    ts = Handle(rk.rk_tableset_destroy, rk.rk_tableset_build(tables))
    s.buf = buf
    s.handle = Handle(rk.rk_batch_destroy, rk.rk_batch_create(
        ts.value, c["items"], int(lens.max()), total, cap), ts)
    s.batch = s.handle.value
    rk.rk_batch_set(s.batch, np.arange(c["items"]),
                    [buf[a:a + n] for a, n in zip(at[:-1], lens)], lens)
    s.out = [torch.as_tensor(_Device(s.handle, ptr, size), device="cuda")
             for ptr, size in zip(rk.rk_batch_results(s.batch), (cap, c["items"] + 1, 2))]
    s.out[0].zero_()


# ------------------------------------------------------------------ one pass

def run(state):
    s, c = state, state.case
    api = c["api"]
    if api == "search":
        rk.rk_search_device(s.table, s.text, c["n"], s.keys, s.cap, s.info, s.ws, s.ws_bytes)
        return s.info, s.keys
    if api == "noalloc":
        rk.rk_search_device_noalloc(s.table, s.text, c["n"], s.keys, s.cap, s.info)
        return s.info, s.keys
    if api == "matcher":
        found = s.matcher.search(s.text)
        s.keys[:found.numel()] = found  # the program's own list, of one size for every text
        return found.numel(), s.keys
    if api == "records":
        _, count = rk.rk_search_device_matches(s.table, s.text, c["n"], s.out, s.cap)
        return count, s.out
    if api == "host":
        _, count = rk.rk_search(s.table, s.text, c["n"], s.keys, s.cap)
        return count, s.keys
    if api == "batch":
        rk.rk_batch_run(s.batch)
        return s.out
    rk.rk_window_hashes_device(s.text, c["n"], c["L"], c["base_log2"], s.out)
    return s.out

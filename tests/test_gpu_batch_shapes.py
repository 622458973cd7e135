"""Batches with the survivor tables in shared memory (s2_in_smem): launch shapes
that fit sets of these sizes, and their matches, whatever the density of the
sets' prefix maps."""

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

from gpu_util import assert_same, require_gpu, to_device  # noqa: E402
from paper_1810_01051_gb300 import rk  # noqa: E402

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def byte_sets(counts, lmin, lmax):
    sets = []
    for k in counts:
        rng = np.random.default_rng(k)
        sets.append([rng.integers(0, 256, int(L), dtype=np.uint8).tobytes()
                     for L in rng.integers(lmin, lmax + 1, k)])
    return sets


# set sizes, lengths, stages, warps, and a tile that fits with every map at one
# slot in two free, or close to that
SHAPES = [
    ((20,), (8, 12), 4, 16, 42848), ((40,), (8, 12), 4, 16, 40544), ((40,), (4, 48), 8, 8, 15936),
    ((5, 30, 64), (4, 48), 8, 8, 13120), ((128,), (4, 48), 8, 8, 5440),
    ((257,), (4, 48), 2, 8, 62784), ((513,), (4, 48), 2, 8, 22848), ((600,), (4, 48), 2, 8, 14912),
]


@pytest.mark.parametrize("counts,lens,stages,warps,tile", SHAPES)
def test_shape_fits_and_matches(counts, lens, stages, warps, tile):
    sets = byte_sets(counts, *lens)
    rng = np.random.default_rng(tile)
    texts = []
    for pats in sets:
        text = rng.integers(0, 256, 200_003, dtype=np.uint8)
        for i, at in enumerate(rng.integers(0, text.size - 64, 400)):
            p = pats[i % len(pats)]
            text[at:at + len(p)] = np.frombuffer(p, np.uint8)
        texts.append(text)
    ts = rk.rk_tableset_build(sets)
    b = rk.rk_batch_create(ts, len(sets), texts[0].size, sum(t.size for t in texts), 1 << 16,
                           warps=warps, tile_bytes=tile, stages=stages, s2_in_smem=1)
    try:
        dev = [to_device(t, 5) for t in texts]
        rk.rk_batch_set(b, np.arange(len(sets)), dev, [t.size for t in texts])
        rk.rk_batch_run(b)
        torch.cuda.synchronize()
        count, status, keys, offsets = rk.rk_batch_read(b, len(sets), 1 << 16)
        assert status == rk.RK_OK and count <= 1 << 16
        info = rk.rk_batch_info(b)
        assert info["s2_in_smem"] == 1 and info["tile_bytes"] == tile
        items, ids, xs = rk.unpack_batch_keys(keys, info["offset_bits"], info["id_bits"])
        for i, (text, pats) in enumerate(zip(texts, sets)):
            a, e = int(offsets[i]), int(offsets[i + 1])
            assert (items[a:e] == i).all()
            assert_same((ids[a:e], xs[a:e]), oracle.rabin_karp(text, pats), f"set {i}")
    finally:
        rk.rk_batch_destroy(b)
        rk.rk_tableset_destroy(ts)


def letter_sets(alphabet, n_sets, k, lmin, lmax):
    rng = np.random.default_rng(n_sets + k)
    sym = np.frombuffer(alphabet, np.uint8)
    return [[rng.choice(sym, int(L)).tobytes() for L in rng.integers(lmin, lmax + 1, k)]
            for _ in range(n_sets)]


@pytest.mark.parametrize("alphabet,k,items,total,ctas", [
    (b"ABCDEFGHIJKLMNOPQRST", 64, 4096, 64 << 20, 3),   # many short texts
    (b"ABCDEFGHIJKLMNOPQRST", 64, 1024, 1 << 30, 3),    # many chunks
    (b"ABCDEFGHIJKLMNOPQRST", 64, 1024, 64 << 20, 1),   # few
    (b"ABCDEFGHIJKLMNOPQRST", 64, 1, 1 << 20, 1),
    (b"ACGT", 256, 4096, 256 << 20, 1),                 # crowds of survivors
    (b"ACGT", 256, 4096, 16 << 20, 3),                  # of very short texts
])
def test_default_shape(alphabet, k, items, total, ctas):
    """The launch shape by the limits and the tables, and with it the matches of
    one text (the texts of a batch may be fewer than its limits)."""
    pats = letter_sets(alphabet, 3, k, 4, 48)
    ts = rk.rk_tableset_build(pats)
    b = rk.rk_batch_create(ts, items, 1 << 20, total, 1 << 20)
    try:
        info = rk.rk_batch_info(b)
        assert info["ctas_per_sm"] == ctas and info["warps"] == (8 if ctas == 3 else 16)
        rng = np.random.default_rng(k)
        text = rng.choice(np.frombuffer(alphabet, np.uint8), 150_001)
        rk.rk_batch_set(b, [1], [to_device(text, 3)], [text.size])
        rk.rk_batch_run(b)
        torch.cuda.synchronize()
        count, status, keys, _ = rk.rk_batch_read(b, 1, 1 << 20)
        assert status == rk.RK_OK and count <= 1 << 20
        _, ids, xs = rk.unpack_batch_keys(keys, info["offset_bits"], info["id_bits"])
        assert_same((ids, xs), oracle.rabin_karp(text, pats[1]), f"{items} {total}")
    finally:
        rk.rk_batch_destroy(b)
        rk.rk_tableset_destroy(ts)

"""Tables of different shared-memory sizes searched from several threads: a
launch limit raised by one thread must hold when another thread's smaller
table sets its own."""

import threading

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

from gpu_util import assert_same, keys_to_pairs, require_gpu, search_table, to_device  # noqa: E402
from paper_1810_01051_gb300 import rk  # noqa: E402

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def test_smaller_table_in_another_thread():
    rng = np.random.default_rng(8)
    text = rng.integers(0, 4, 300_001, dtype=np.uint8) + ord("a")
    # the same kernel (step 2, tables in shared memory) at two sizes
    small = [b"abcda", b"bcddab"]
    large = [bytes(text[i * 40:i * 40 + 5 + i % 30].tolist()) for i in range(90)]
    tables = {"small": rk.rk_build(small), "large": rk.rk_build(large)}
    info = {n: rk.rk_table_info(t) for n, t in tables.items()}
    assert info["small"]["smem_bytes"] < info["large"]["smem_bytes"]
    assert info["small"]["role_step"] == info["large"]["role_step"] == 2
    d = to_device(text)
    got = {}

    def search(name):
        keys, count, status = search_table(tables[name], d, text.size, 1 << 17)
        got[name] = (status, keys_to_pairs(keys[:count]))

    search("large")
    t = threading.Thread(target=search, args=("small",))
    t.start()
    t.join()
    search("large")
    for name, pats in (("small", small), ("large", large)):
        assert got[name][0] == rk.RK_OK
        assert_same(got[name][1], oracle.rabin_karp(text, pats), name)
    for t in tables.values():
        rk.rk_destroy(t)

"""A search given room for a candidate list completes its survivors in the scan
or lists them, by table and text size: on both sides of the size where that
changes, and for every kind of table, its output is the one of the listed scan
(rk_scan_device_ws, always listed) and of the scan without a list."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from gpu_util import require_gpu  # noqa: E402
from paper_1810_01051_gb300 import rk  # noqa: E402

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


MIB = 1 << 20
# shortest pattern, patterns, options, the size where the route changes
TABLES = {
    "roles": (7, 60, dict(), 48 * MIB),
    "roles, tables in L2": (7, 1500, dict(), 48 * MIB),
    "sampled": (7, 60, dict(role_step=1), 4 * MIB),
    "sampled, tables in L2": (7, 1500, dict(role_step=1), 4 * MIB),
    "prefix": (7, 60, dict(role_step=1, sample=1), 4 * MIB),
    "short prefix": (3, 60, dict(), 48 * MIB),
    "no filter": (7, 60, dict(filter=rk.RK_FILTER_NONE), 4 * MIB),
}


@pytest.mark.parametrize("name", sorted(TABLES))
def test_routes_agree(name):
    lmin, k, opts, LINE = TABLES[name]
    g = torch.Generator(device="cuda").manual_seed(len(name))
    buf = torch.randint(97, 123, (LINE + 32,), generator=g, device="cuda", dtype=torch.uint8)
    rng = np.random.default_rng(len(name))
    pats = []
    host = buf.cpu().numpy()
    for i in range(k):
        at, L = int(rng.integers(0, LINE - 64)), lmin + i % 23
        p = host[at:at + L].tobytes()
        pats.append(p)
        for at in rng.integers(0, LINE - 64, 20):
            host[at:at + L] = np.frombuffer(p, np.uint8)
    buf.copy_(torch.from_numpy(host))
    tail = torch.tensor(list(pats[0]), dtype=torch.uint8, device="cuda")
    table = rk.rk_build(pats, **opts)
    try:
        for n, mis in ((LINE - 1, 3), (LINE, 0), (LINE + 1, 9)):
            text = buf[mis:mis + n]
            text[n - tail.numel():] = tail
            cap = 1 << 20
            sort_bytes = rk.rk_workspace_bytes(table, cap)
            list_bytes = rk.rk_scan_workspace_bytes(table, n)
            results = []
            for route in ("search", "listed", "in scan"):
                d = torch.zeros(cap, dtype=torch.int64, device="cuda")
                info = torch.zeros(2, dtype=torch.int64, device="cuda")
                ws = torch.full((sort_bytes + list_bytes,), 0xA5, dtype=torch.uint8, device="cuda")
                if route == "search":
                    rk.rk_search_device(table, text, n, d, cap, info, ws, sort_bytes + list_bytes)
                elif route == "listed":
                    rk.rk_scan_device_ws(table, text, n, d, cap, info, ws[sort_bytes:], list_bytes)
                    rk.rk_sort_device(table, n, d, cap, info, ws, sort_bytes)
                else:
                    rk.rk_scan_device(table, text, n, d, cap, info)
                    rk.rk_sort_device(table, n, d, cap, info, ws, sort_bytes)
                torch.cuda.synchronize()
                assert int(info[1]) == rk.RK_OK
                results.append(d[:int(info[0])].cpu().numpy())
            assert results[0].size >= k
            assert np.array_equal(results[0], results[1]), (n, mis)
            assert np.array_equal(results[0], results[2]), (n, mis)
    finally:
        rk.rk_destroy(table)

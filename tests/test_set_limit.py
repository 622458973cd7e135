"""The largest pattern set a table takes, on CPU: the rule's header is host-only
C++, compiled here with g++ (tests/limit_check.cpp), and a table's own size stays
within what the rule says it may exceed the counted one by."""

import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1810_01051_gb300 import rk

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1810_01051_gb300", "csrc")


def test_limit(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not found")
    exe = tmp_path / "limit_check"
    subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-Werror", f"-I{CSRC}",
                    os.path.join(ROOT, "tests", "limit_check.cpp"), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr


def counted(pats, info):
    """set_bytes of a set, and the prefix bit set, from the patterns."""
    part = lambda n: -(-n // 256) * 256  # noqa: E731
    pow2 = lambda x: 1 << max(0, int(x - 1).bit_length())  # noqa: E731
    q = info["gram_len"]
    by_len = {}
    for p in pats:
        by_len.setdefault(len(p), set()).add(p)
    slots = sum(max(2, pow2(2 * len(v))) for v in by_len.values())
    samp = 0
    if info["sample_step"] == 4:
        samp = max(16, pow2(2 * len({p[j:j + 4] for p in pats for j in range(4)})))
    k = len(pats)
    parts = [16 * max(16, pow2(2 * info["n_grams"])), 4 * len({(p[:q], len(p)) for p in pats}) + 4,
             8 * (info["max_len"] + 1), 16 * slots + 16, 4 * k + 4,
             sum(-(-len(p) // 8) * 8 for p in pats) + 16, 8 * k + 8, 4 * k + 4,
             4 * info["n_lengths"] + 4, 8 * samp + 8]
    return sum(map(part, parts)) + part(info["filter_smem_bytes"] + 16)


@pytest.mark.parametrize("k,lmin,lmax", [(5, 8, 8), (300, 7, 40), (3000, 1, 6), (20_000, 8, 64)])
def test_table_size_against_the_count(k, lmin, lmax):
    rng = np.random.default_rng(k)
    pats = [rng.integers(0, 256, int(L), dtype=np.uint8).tobytes()
            for L in rng.integers(lmin, lmax + 1, k)]
    for role_step in (1, 0):
        info = rk.rk_plan(pats, role_step=role_step)
        filters = (1 << 20) if info["role_step"] or info["sample_step"] == 4 else 512
        over = info["device_bytes"] - counted(pats, info)
        assert 0 <= over <= 12 * k + (32 << 20) + filters

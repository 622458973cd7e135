"""Which sets have their survivor tables copied to shared memory (rk_plan, no
GPU): the prefix map's density gives way before the copy does, and a table
without a prefilter carries no map in the copy."""

import numpy as np
import pytest

from paper_1810_01051_gb300 import rk

CASES = [
    # lengths, options, pattern counts whose tables fit with the densest map
    ((8, 64), {}, (100, 256, 288, 312)),
    ((25, 800), {}, (64, 72)),
    ((8, 64), dict(role_step=1), (72, 112, 312, 336)),
    ((8, 8), dict(role_step=1), (72, 112, 504, 512)),
    ((16, 16), dict(filter=rk.RK_FILTER_FLAT), (256, 264, 504)),
    ((4, 32), dict(filter=rk.RK_FILTER_NONE), (512, 520, 700)),
    ((8, 64), dict(stages=3), (312,)),
]


@pytest.mark.parametrize("lens,opts,counts", CASES)
def test_copied(lens, opts, counts):
    for k in counts:
        rng = np.random.default_rng(k * 7 + lens[0])
        pats = [rng.integers(0, 256, int(L), dtype=np.uint8).tobytes()
                for L in rng.integers(lens[0], lens[1] + 1, k)]
        info = rk.rk_plan(pats, **opts)
        assert info["s2_smem_bytes"] > 0, k
        assert info["smem_bytes"] <= rk.GB300_SMEM_OPTIN - 1024
        # one slot in two of the map is free at least: 16 bytes a slot
        if "filter" not in opts:
            assert info["s2_smem_bytes"] >= 32 * info["n_grams"]

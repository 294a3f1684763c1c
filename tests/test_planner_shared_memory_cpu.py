"""The resident CTAs that a pair-kernel plan counts on fit the SM's shared memory: 228 KB,
of which each CTA takes its dynamic part (column arrays, per-warp space), its static
arrays and 1 KB."""
import numpy as np
import pytest

import __graft_entry__
from paper_2402_16712_gb300 import l1line

STATIC = 32 * 56 + 16  # 32 per-penalty thresholds and the counters


@pytest.fixture(scope="module", autouse=True)
def _lib():
    __graft_entry__.build()
    l1line.load()


@pytest.mark.parametrize("m", [20, 2000])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_planned_ctas_fit(dtype, m):
    size = np.dtype(dtype).itemsize
    for n in range(128, l1line.max_rows(dtype) + 1, 128):
        p = l1line.plan_for(dtype, n, m, 152)
        column = (n * size if p["column"] == 1 else 0) + 2 * 4 * n + 128
        warp = 1024 + 6 * min(n, 128)
        need = column + p["warps"] * warp + STATIC + 1024
        assert need * p["ctas_per_sm"] <= 228 * 1024, (n, p)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_limit_on_rows_does_not_depend_on_the_type(dtype):
    assert l1line.max_rows(dtype) == 20608


def test_a_callers_shape_beyond_that_is_still_taken():
    l1line.set_tuning({"warps": 15, "ctas_per_sm": 2})
    try:
        p = l1line.plan_for(np.float32, 7296, 512, 152)
    finally:
        l1line.set_tuning(None)
    assert (p["warps"], p["ctas_per_sm"]) == (15, 2)

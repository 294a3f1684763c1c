"""The global-memory path's bracket search against the oracle where its steps
can go wrong: row counts around its vectors, slices and clusters, weights so
uneven that the sample misses, penalties that put the median at 0, columns with
few valid rows, ratios closer together than its bins, and ties.  Every v bit
for bit, s and z within the bar of tests/_parity.py."""
import numpy as np
import pytest
import torch

from paper_2402_16712_gb300 import l1line
from tests._parity import check_scan

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _rows(dtype):
    n = l1line.max_rows(dtype)
    return [n + 1, n + 129, 65535, 65536, 65537, 131075]


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("which", range(6))
def test_row_counts(which, dtype):
    n = _rows(dtype)[which]
    rng = np.random.default_rng(n)
    X = rng.normal(size=(n, 3)).astype(dtype)
    check_scan(X, [0.0, 0.01 * n, 2.0 * n], where=f"n={n}")


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("kind", ["weights", "sparse", "close", "ties", "signs"])
def test_what_the_sample_does_not_show(kind, dtype):
    n = 70001
    rng = np.random.default_rng(6)
    x = rng.normal(size=n)
    if kind == "weights":  # a few rows hold most of the weight, rows in runs
        x = x * np.exp(3.0 * np.sin(np.arange(n) / 900.0)) * rng.lognormal(0, 2, size=n)
        X = np.stack([x, 0.5 * x + rng.normal(size=n), rng.standard_t(1.2, size=n)], axis=1)
    elif kind == "sparse":
        X = rng.normal(size=(n, 3)) * (rng.random(size=(n, 3)) < [0.1, 0.5, 1.0])
    elif kind == "close":  # ratios within a few keys of 2, and within 1e-4
        X = np.stack([x, 2.0 * x * (1 + 1e-7 * rng.normal(size=n)),
                      2.0 * x * (1 + 1e-4 * rng.normal(size=n))], axis=1)
    elif kind == "ties":
        X = np.round(2.0 * rng.normal(size=(n, 3)))
    else:  # the median next to and at 0
        X = np.stack([np.abs(x), x - 0.001, np.where(rng.random(n) < 0.6, 0.0, x)], axis=1)
    check_scan(np.ascontiguousarray(X.astype(dtype)), [0.0, 1.0, 1e4], where=kind)

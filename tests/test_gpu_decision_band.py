"""Decisions next to the edge of the 32-bit weights' certainty band: the rows below and
above the crossing weigh the same but for one row, whose weight runs from far below the
truncation of one row to above that of all rows together.

Bar: v, s and z as in tests/_parity.py."""
import numpy as np
import pytest

from tests._parity import check_scan

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _balanced(half, tiny, spread, dtype, seed):
    """Column 0: `half` weights, the same again and one of size `tiny` times the largest;
    the others: ratios to column 0 that put the first half below, the second above, and
    the odd row between, below or above."""
    rng = np.random.default_rng(seed)
    w = np.abs(rng.normal(size=half)) * 2.0 ** rng.uniform(-spread, 0, half)
    w = np.concatenate([w, rng.permutation(w), [tiny * w.max()]]) * rng.choice([-1, 1], 2 * half + 1)
    b = w.astype(dtype)
    cols = [b]
    for c in range(5):
        r = np.concatenate([rng.uniform(0.5, 1, half), rng.uniform(2, 3, half), [[1.5, 0.25, 4][c % 3]]])
        cols.append((b * (r if c < 3 else -r).astype(dtype)).astype(dtype))
    X = np.stack(cols, axis=1)
    return np.ascontiguousarray(X[rng.permutation(2 * half + 1)])


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("spread", [0, 12])
@pytest.mark.parametrize("half", [20, 64, 700])
def test_balanced_columns(half, spread, dtype):
    for i, e in enumerate([-52, -44, -36, -32, -30, -28, -26, -24, -22, -20, -16]):
        X = _balanced(half, 2.0 ** e, spread, dtype, 10 * half + i)
        check_scan(X, np.array([0.0, 2.0 ** (e - 1)]), where=f"{half} {spread} {e}")

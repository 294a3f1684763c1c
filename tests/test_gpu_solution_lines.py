"""The solution path of data whose ratios differ in the last place only (rounded
measurements and multiples of one column, in double): a change of v that leaves intercept
and slope as they are is no piece, so no two neighbours are the same line."""
import numpy as np
import pytest
import torch

from paper_2402_16712_gb300 import l1line

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("kind", ["tenths", "multiples"])
@pytest.mark.parametrize("m", [1, 2, 12])
def test_no_piece_repeats_its_line(kind, m):
    n = 300
    rng = np.random.default_rng(2)
    t = rng.normal(size=(n, 1))
    if kind == "tenths":
        X = np.round(t * rng.uniform(0.2, 1.2, (1, m)) + 0.3 * rng.normal(size=(n, m)), 1)
    else:
        X = t * rng.integers(1, 9, (1, m)) / 2
    st, jh, ic, sl, v = l1line.solution_path(torch.from_numpy(np.ascontiguousarray(X)).cuda())
    assert bool((st[1:] > st[:-1]).all())
    same = (jh[1:] == jh[:-1]) & (ic[1:] == ic[:-1]) & (sl[1:] == sl[:-1])
    assert not bool(same.any())

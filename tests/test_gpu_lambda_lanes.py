"""A batch of penalties, decided one per lane, against one scan per penalty at
the counts around a warp's 32 lanes and a launch's limits: v and s bit for bit
(the same medians, and the same residual sum of each), with equal penalties, 0
and penalties beyond every column's weight among them, in any order."""
import numpy as np
import pytest
import torch

from paper_2402_16712_gb300 import datagen, l1line

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("kind", ["planted", "integers"])
@pytest.mark.parametrize("nl", [3, 8, 31, 32, 33, 65, 257])
def test_lambdas_match_single_scans(nl, kind, dtype):
    if kind == "planted":
        X, _, _ = datagen.planted(datagen.Planted(300, 9, 3, 0.1, 0.1, 5.0, nl, dtype))
    else:
        X = datagen.small_integers(150, 9, nl, lo=-4, hi=4, zero_frac=0.2, dtype=dtype)
    X = torch.from_numpy(np.ascontiguousarray(X)).cuda()
    rng = np.random.default_rng(nl)
    lams = np.concatenate([[0.0, 1e9, 2.0], 10.0 ** rng.uniform(-3, 4, nl)])[:nl]
    lams[nl // 2] = lams[nl - 1]
    rng.shuffle(lams)
    v, s, z, ws = l1line.scan(X, lams)
    assert l1line.status(ws) == l1line.OK
    for t in sorted({0, 1, 2, nl // 2, nl - 1, *rng.integers(0, nl, 12).tolist()}):
        v1, s1, z1, _ = l1line.scan(X, [lams[t]])
        assert torch.equal(v[t], v1[0]) and torch.equal(s[t], s1[0]) and torch.equal(z[t], z1[0])

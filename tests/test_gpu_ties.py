"""Tied and nearly tied ratios in the pair kernels: rounded data, counts, sparse
columns, columns that are (nearly) multiples of one another, at the rows around a
128-row group and beyond a warp's lanes, with one penalty and with batches below and
from 16 on.

Bar: v, s and z as in tests/_parity.py.  A fit of such data in double takes at most 20
times as long as one of continuous data (it takes up to 6; where every such pair went to
the exact search, 100 to 300)."""
import numpy as np
import pytest
import torch

from paper_2402_16712_gb300 import l1line
from tests._parity import assert_v_equal, check_scan

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _data(kind, n, m, dtype, seed=1):
    rng = np.random.default_rng(seed)
    t = rng.normal(size=(n, 1))
    if kind == "continuous":
        X = t * rng.uniform(0.2, 1.2, (1, m)) + 0.3 * rng.normal(size=(n, m))
    elif kind == "ints":
        X = rng.integers(1, 6, (n, m))
    elif kind == "signed":
        X = rng.integers(-3, 4, (n, m))
    elif kind == "sparse":
        X = rng.normal(size=(n, m)) * (rng.random((n, m)) > 0.9)
    elif kind == "tenths":
        X = np.round(t * rng.uniform(0.2, 1.2, (1, m)) + 0.3 * rng.normal(size=(n, m)), 1)
    elif kind == "near":
        X = (t + 3) * rng.uniform(0.5, 1.5, (1, m)) * (1 + 1e-5 * rng.normal(size=(n, m)))
    elif kind == "nearer":
        X = (t + 3) * rng.uniform(0.5, 1.5, (1, m)) * (1 + 1e-8 * rng.normal(size=(n, m)))
    else:  # multiples
        X = t * rng.integers(1, 9, (1, m)) / 2
    return np.ascontiguousarray(np.asarray(X, dtype=np.float64).astype(dtype))


KINDS = ["ints", "signed", "sparse", "tenths", "near", "nearer", "multiples"]


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n,nl", [(33, 1), (128, 4), (129, 1), (700, 17), (2000, 1), (2000, 4),
                                  (5000, 1)])
def test_ties_match_oracle(n, nl, kind, dtype):
    X = _data(kind, n, 6, dtype)
    lams = np.array([0.4]) if nl == 1 else np.concatenate([[0.0], np.logspace(-3, 0.5, nl - 1)])
    check_scan(X, lams * n / 50, where=f"{kind} {n} {nl}")


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("nl", [1, 5, 20])
def test_tied_batches_match_single_scans(nl, dtype):
    Xs = [_data(k, n, 5, dtype, n) for k, n in zip(KINDS, (100, 300, 150, 700, 90, 1500, 40))]
    lams = [np.logspace(-2, 1, nl) * len(X) / 50 for X in Xs]
    Xd = [torch.from_numpy(X).cuda() for X in Xs]
    bat = l1line.Batched(Xd, lams)
    bat.run()
    assert bat.status() == l1line.OK
    for X, lam, (v, obj, js) in zip(Xd, lams, bat.results()):
        v1, s1, z1, _ = l1line.scan(X, lam)
        for t in range(nl):
            j = int(z1[t].argmin())
            assert int(js[t]) == j and float(obj[t]) == float(z1[t, j])
            assert_v_equal(v[t].cpu().numpy(), v1[t, j].cpu().numpy())


@pytest.mark.parametrize("kind", ["ints", "signed", "sparse", "near"])
def test_ties_take_no_exact_search(kind):
    us = []
    for k in ("continuous", kind):
        X = torch.from_numpy(_data(k, 2000, 64, "float64")).cuda()
        ws = l1line.Workspace.for_shape(X.dtype, 2000, 64, 1)
        t = []
        for _ in range(5):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            l1line.fit(X, [20.0], workspace=ws)
            e1.record()
            e1.synchronize()
            t.append(e0.elapsed_time(e1))
        assert l1line.status(ws) == l1line.OK
        us.append(min(t[1:]))
    assert us[1] <= 20 * us[0]

"""Residuals of the penalty paths' entries (l1line_path_write's out_resid) and
the paths at the edges of the kernels' steps (128 rows, a queue of 32, sorts of
64 and more), against exact rational sums and the oracle.

Bar: with C = sum_i |x_ik|, R(t) is C - 2 B + t (2 S - Q), each term at most C
and rounded to double (2^-53), the fixed-point sums short of less than n
2^-60 C: |R - exact| <= 2^-50 C + n 2^-58 C."""
from fractions import Fraction

import numpy as np
import pytest
import torch

import oracle
from paper_2402_16712_gb300 import datagen, l1line

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _check(X):
    n, m = X.shape
    off, lam, v, ln, ws, res = l1line.paths(torch.from_numpy(X).cuda(), residuals=True)
    assert l1line.status(ws) == l1line.OK
    off, lam, v, ln, res = (t.cpu().numpy() for t in (off, lam, v, ln, res))
    F = [[Fraction(float(x)) for x in X[:, k]] for k in range(m)]
    for j in range(m):
        for k in range(m):
            p = j * m + k
            o, L = off[p], int(ln[p])
            rl, rv = oracle.path(X, j, k)
            assert L == rl.size and np.array_equal(v[o:o + L], rv.astype(X.dtype))
            C = sum(abs(x) for x in F[k])
            tol = C * (Fraction(1, 2 ** 50) + Fraction(n, 2 ** 58))
            for g in sorted({0, 1, L // 2, L - 2, L - 1} & set(range(L))):
                t = Fraction(float(v[o + g]))
                want = sum(abs(x - t * b) for x, b in zip(F[k], F[j]))
                assert abs(Fraction(float(res[o + g])) - want) <= tol, (j, k, g, L)


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("n", [1, 31, 32, 127, 128, 129, 300, 1025])
def test_residuals_over_row_counts(n, dtype):
    X, _, _ = datagen.planted(datagen.Planted(n, 5, 2, 0.1, 0.1, 5.0, n, dtype))
    _check(np.ascontiguousarray(X))


@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_residuals_many_rows_in_range_ties_and_zeros(dtype):
    rng = np.random.default_rng(3)
    x0 = rng.normal(size=700)
    X = np.stack([x0, 2 * x0 + 0.01 * rng.normal(size=700), np.round(3 * x0),
                  np.round(rng.normal(size=700)), np.zeros(700)], axis=1)
    _check(np.ascontiguousarray(X[:, :4].astype(dtype)))
    _check(np.ascontiguousarray(X[:140].astype(dtype)))


@pytest.mark.parametrize("scale", [(1e-40, 1e-38, 1e-36, 1e-39), (1e38, 3e36, 1e38, 1e37)])
def test_residuals_of_magnitudes_beyond_the_approximate_keys(scale):
    # subnormal and huge columns: every row is divided
    rng = np.random.default_rng(4)
    X = rng.uniform(-1, 1, size=(200, 4)) * np.array(scale)
    _check(np.ascontiguousarray(X.astype(np.float32)))


def test_residuals_of_a_column_beyond_the_fixed_point():
    # one row 2^40 or 2^28 above the others: the fixed point drops the others' low bits
    rng = np.random.default_rng(5)
    X = rng.uniform(-1, 1, size=(1030, 4))
    X[17, 1] = 2.0 ** 40
    X[19, 2] = -2.0 ** 28
    _check(np.ascontiguousarray(X.astype(np.float32)))

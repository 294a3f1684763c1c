"""The certainty band of the 32-bit weights, replayed in whole numbers: for every set of
rows the true 2S - Q lies within e of the truncated one, with e from the 64-bit and the
32-bit total as the pair kernel takes it, and e is no more than a unit per row and one."""
from fractions import Fraction

import numpy as np
import pytest


@pytest.mark.parametrize("seed", range(40))
def test_true_difference_lies_inside(seed):
    rng = np.random.default_rng(seed)
    n = int(rng.integers(2, 60))
    w = np.abs(rng.normal(size=n)) * 2.0 ** rng.uniform(-40 * (seed % 3), 0, n)
    if seed % 2:
        w = w.astype(np.float32).astype(np.float64)
    if seed % 5 == 0:  # remainders close to one unit
        w = (np.floor(w * 2.0 ** 20) + 1 - 2.0 ** -20) * 2.0 ** -20
    sigma = 60 - int(np.floor(np.log2(w.max()))) - n.bit_length()
    true = [Fraction(float(x)) * Fraction(2) ** sigma for x in w]
    q = [int(x) for x in true]
    inexact = sum(a != b for a, b in zip(q, true))
    Q = sum(q)
    shift = 0
    while sum(x >> shift for x in q) >= 1 << 32:
        shift += 1
    q32 = [x >> shift for x in q]
    Q32 = sum(q32)
    e = ((Q + inexact) >> shift) + 1 - Q32
    unit = [x / (1 << shift) for x in true]
    rem = [u - a for u, a in zip(unit, q32)]
    order = np.argsort([float(r) for r in rem])
    sets = [order[:k] for k in range(n + 1)] + [order[k:] for k in range(n + 1)]
    sets += [np.flatnonzero(rng.random(n) < 0.5) for _ in range(50)]
    for s in sets:
        D = 2 * sum(q32[i] for i in s) - Q32
        D_true = 2 * sum(unit[i] for i in s) - sum(unit)
        assert D - e < D_true < D + e
    assert e <= n + 1

"""The exact path's pairs are spread over all SMs however its kernel is launched:
behind the pair kernel, beside whose last CTAs it is placed, or behind the kernel
for more rows than that takes, which it waits for.  The same pairs with 1% more
rows behind the latter may not be much faster (bar: 1.6 times; on a few SMs the
first took 2 to 4 times as long)."""
import pytest
import torch

from paper_2402_16712_gb300 import l1line

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("m", [24, 48])
def test_exact_pairs_take_every_sm(m):
    rows = l1line.max_rows(torch.float64)
    best = []
    for n in (rows, rows + 128):
        g = torch.Generator(device="cuda").manual_seed(m)
        X = torch.randn(n, m, generator=g, device="cuda", dtype=torch.float64)
        ws = l1line.Workspace.for_shape(X.dtype, n, m, 1)
        ms = []
        for _ in range(4):
            t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            t0.record()
            l1line.scan(X, [0.5], workspace=ws, flags=l1line.FLAG_FORCE_EXACT)
            t1.record()
            t1.synchronize()
            ms.append(t0.elapsed_time(t1))
        assert l1line.status(ws) == l1line.OK
        best.append(min(ms[1:]))
    assert best[0] <= 1.6 * best[1]

"""The chain of short kernels of a fit, placed ahead of each other's end: back to
back on one workspace, on two streams, captured in a graph, and with the fused
last step at the sizes around its limit (jhat x columns = 4096).

Bar: bit for bit the same as fits with a synchronisation after each, and jhat*
the smallest index of the smallest z of a scan."""
import numpy as np
import pytest
import torch

from paper_2402_16712_gb300 import datagen, l1line

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _data(n, m, seed, dtype):
    X, _, _ = datagen.planted(datagen.Planted(n, m, max(1, m // 8), 0.1, 0.1, 5.0, seed, dtype))
    return torch.from_numpy(np.ascontiguousarray(X)).cuda()


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("n,m", [(40, 1), (200, 20), (90, 63), (90, 64), (90, 65)])
def test_back_to_back_fits(n, m, dtype):
    Xs = [_data(n, m, s, dtype) for s in range(6)]
    want = []
    for X in Xs:
        v, obj, js, ws = l1line.fit(X, [0.1, 2.0])
        torch.cuda.synchronize()
        assert l1line.status(ws) == l1line.OK
        z = l1line.scan(X, [0.1, 2.0])[2].cpu().numpy()
        assert np.array_equal(js.cpu().numpy(), z.argmin(axis=1))
        assert np.array_equal(obj.cpu().numpy(), z.min(axis=1))
        want.append((v.cpu(), obj.cpu(), js.cpu()))
    ws = l1line.Workspace.for_shape(Xs[0].dtype, n, m, 2)
    side = torch.cuda.Stream()
    ws2 = l1line.Workspace.for_shape(Xs[0].dtype, n, m, 2)
    torch.cuda.synchronize()
    got = []
    for r in range(5):
        for i, X in enumerate(Xs):
            got.append((i, l1line.fit(X, [0.1, 2.0], workspace=ws)))
            with torch.cuda.stream(side):
                got.append((i, l1line.fit(X, [0.1, 2.0], workspace=ws2, stream=side)))
    torch.cuda.synchronize()
    for i, o in got:
        assert all(torch.equal(a.cpu(), b) for a, b in zip(o[:3], want[i]))


def test_captured_chain():
    X = _data(200, 20, 3, "float64")
    v, obj, js, ws = l1line.fit(X, [0.1])
    want = [t.clone() for t in (v, obj, js)]
    out = tuple(torch.zeros_like(t) for t in want)
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        for _ in range(3):
            l1line.fit(X, [0.1], workspace=ws, out=out, stream=torch.cuda.current_stream())
    for _ in range(4):
        for t in out:
            t.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(out, want))


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("m", [1, 3, 4, 15, 16])
@pytest.mark.parametrize("offset", [0, 1])
def test_narrow_staging(m, dtype, offset):
    # the contiguous staging of up to 16 columns: X aligned to 16 bytes or not,
    # a last CTA of a few rows; against the same rows as 17 columns (the other)
    n = 152 * 256 + 3
    g = torch.Generator(device="cuda").manual_seed(m)
    flat = torch.randn(n * m + 1, generator=g, device="cuda", dtype=dtype)
    X = flat[offset:offset + n * m].view(n, m)
    W = torch.zeros((n, 17), device="cuda", dtype=dtype)
    W[:, :m] = X
    v, s, z, ws = l1line.scan(X, [0.5])
    assert l1line.status(ws) == l1line.OK
    vw, sw, zw, _ = l1line.scan(W, [0.5])
    assert torch.equal(v, vw[:, :m, :m]) and torch.equal(s, sw[:, :m, :m])
    X[n - 1, m - 1] = float("inf")
    assert l1line.status(l1line.scan(X, [0.5])[3]) != l1line.OK


@pytest.mark.parametrize("n_inst", [3, 305])
def test_rank_loss_lengths(n_inst):
    # one row, an empty instance, a cluster's 1024 rows and a row more, and more
    # than a thread keeps; double reference, float outputs
    lens = np.resize([1, 0, 1024, 1025, 127, 4097, 8193], n_inst)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    rng = np.random.default_rng(n_inst)
    s, t = (rng.normal(0, 3, size=off[-1]).astype(np.float32) for _ in range(2))
    loss, ds = l1line.rank_loss(torch.from_numpy(s).cuda(), torch.from_numpy(t).cuda(),
                                torch.from_numpy(off).cuda())
    loss, ds = loss.cpu().numpy(), ds.cpu().numpy()
    for b in range(n_inst):
        x, u = (a[off[b]:off[b + 1]].astype(np.float64) for a in (s, t))
        if not len(x):
            assert loss[b] == 0.0
            continue
        p, q = np.exp(x - x.max()), np.exp(u - u.max())
        L = x.max() + np.log(p.sum()) - (q * x).sum() / q.sum()
        p, q = p / p.sum(), q / q.sum()
        assert abs(loss[b] - L) <= 2.0 ** -23 * max(1.0, abs(L))
        want = (p - q) / n_inst
        assert np.all(np.abs(ds[off[b]:off[b + 1]] - want) <=
                      2.0 ** -23 * np.abs(want) + 2.0 ** -40 * (p + q) / n_inst)

"""The solution path from given pair paths (l1line_solution_path) against a
numpy evaluation of the functions it takes the minimum of: none of them
dropped (all nearly equal), most of them dropped, more equal lambdas than one
bucket of the sort ranks, lambdas over 15 decades, one column, no changes.

Bar: every sum here has at most m terms of size z, in double on both sides:
|z*(lambda) - min_j z_j(lambda)| <= (m + 8) 2^-52 of the largest z, plus the
1e-12 relative within which two functions count as equal."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2402_16712_gb300 import l1line

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _functions(m, L, spread, lams, dtype, seed):
    """Pair paths: v falls to 0 in L - 1 steps at rising lambdas and R rises so
    that R + lambda |v| is continuous (hence concave); every jhat's values at 0
    and beyond the last lambda agree up to `spread`."""
    rng = np.random.default_rng(seed)
    off, lam, v, res, ln = [0], [], [], [], []
    for j in range(m):
        for k in range(m):
            if k == j:
                lam.append([0.0]), v.append([1.0]), res.append([0.0])
            else:
                s = rng.exponential(size=L - 1).astype(dtype)
                if lams == "ties":
                    q = np.repeat([0.5, 2.0], [(L - 1) // 2, L - 1 - (L - 1) // 2])
                elif lams == "wide":
                    q = np.sort(10.0 ** rng.uniform(-12, 3, size=L - 1))
                else:
                    q = np.sort(rng.uniform(0, 10, size=L - 1))
                vv = np.append(np.cumsum(s[::-1].astype(np.float64))[::-1], 0.0).astype(dtype)
                sg = rng.choice([-1.0, 1.0])
                d = q * (vv[:-1].astype(np.float64) - vv[1:].astype(np.float64))
                top = 50.0 * L * (1.0 + spread * rng.uniform())
                r = top - np.append(np.cumsum(d[::-1])[::-1], 0.0)
                lam.append(np.append(0.0, q)), v.append(sg * vv), res.append(r)
            ln.append(len(lam[-1]))
            off.append(off[-1] + ln[-1])
    cat = lambda x, t: np.concatenate([np.asarray(a, dtype=t) for a in x])
    return (np.array(off, dtype=np.int64), cat(lam, np.float64), cat(v, dtype),
            cat(res, np.float64), np.array(ln, dtype=np.int32))


def _value(m, off, lam, v, res, ln, q):
    z = np.zeros(m)
    for j in range(m):
        for k in range(m):
            o, n = off[j * m + k], ln[j * m + k]
            e = o + np.searchsorted(lam[o:o + n], q, side="right") - 1
            z[j] += res[e] + q * abs(float(v[e]))
    return z


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("m,L,spread,lams", [
    (1, 1, 0.0, "even"), (2, 1, 0.0, "even"), (2, 2, 0.0, "even"), (5, 40, 0.0, "even"),
    (33, 20, 0.0, "even"), (33, 20, 1.0, "even"), (12, 60, 0.0, "wide"),
    (3, 1500, 0.0, "ties"), (4, 1025, 0.0, "ties")])
def test_minimum_of_given_functions(m, L, spread, lams, dtype):
    off, lam, v, res, ln = _functions(m, L, spread, lams, dtype, 7 * m + L)
    d = [torch.from_numpy(x).cuda() for x in (off, lam, v, res, ln)]
    entries = int(off[-1])
    cap = entries + 8
    lib = l1line.load()
    ws = l1line.Workspace(int(lib.l1line_solution_path_workspace_bytes(m, entries)))
    st, ic, sl = (torch.zeros(cap, dtype=torch.float64, device="cuda") for _ in range(3))
    jh = torch.zeros(cap, dtype=torch.int32, device="cuda")
    vs = torch.zeros((cap, m), dtype=d[2].dtype, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    f = lib.l1line_solution_path_f32 if dtype == np.float32 else lib.l1line_solution_path_f64
    rc = f(m, *[x.data_ptr() for x in d], entries, st.data_ptr(), jh.data_ptr(), ic.data_ptr(),
           sl.data_ptr(), vs.data_ptr(), cnt.data_ptr(), cap, ctypes.c_void_p(ws.ptr), ws.nbytes,
           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == l1line.OK and l1line.status(ws) == l1line.OK
    c = int(cnt.item())
    assert 1 <= c <= cap
    st, jh, ic, sl, vs = (x[:c].cpu().numpy() for x in (st, jh, ic, sl, vs))
    assert st[0] == 0.0 and np.all(np.diff(st) > 0)
    top = float(lam.max())
    rng = np.random.default_rng(1)
    qs = np.concatenate([rng.uniform(0, 1.2 * top + 1, 40), 10.0 ** rng.uniform(-12, 1, 20),
                         (0.5 * (st[:-1] + st[1:]))[:: max(1, c // 40)]])
    for q in qs:
        z = _value(m, off, lam, v, res, ln, q)
        e = int(np.searchsorted(st, q, side="right")) - 1
        tol = ((m + 8) * 2.0 ** -52 + 2e-12) * np.abs(z).max()
        if lams == "wide":
            tol += 1e-12 * q * sl.max()
        if dtype == np.float32:  # the v of a step are rounded: its two sides meet to 2^-24
            tol += 2.0 ** -22 * q * sl.max()
        assert abs(ic[e] + sl[e] * q - z.min()) <= tol, (q, e, ic[e] + sl[e] * q, z.min())
        assert z[jh[e]] - z.min() <= tol
        j = int(jh[e])
        for k in range(m):
            o, n = off[j * m + k], ln[j * m + k]
            assert vs[e, k] == v[o + np.searchsorted(lam[o:o + n], st[e], side="right") - 1]

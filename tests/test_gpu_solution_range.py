"""Algorithm 3 at the ends of the doubles' range: residuals whose first and last add up
beyond it although every objective is finite, subnormal ones, and ones that are not finite
(status L1L_ERR_NONFINITE, not a plausible line).

Bar: |z* - min_j z_j| <= (m + 8) 2^-52 z plus the 1e-12 relative within which two
functions count as equal, plus m + 8 units of the smallest subnormal."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2402_16712_gb300 import l1line

pytestmark = pytest.mark.gpu
M = 4


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _paths(top, lam_scale):
    """M functions of three entries per pair, residuals 0.8, 0.9 and 1 times top."""
    off, lam, v, res, ln = [0], [], [], [], []
    for j in range(M):
        for k in range(M):
            own = j == k
            lam.append([0.0] if own else [0.0, lam_scale, 2.0 * lam_scale])
            v.append([1.0] if own else [1.5 + 0.1 * j, 0.5, 0.0])
            res.append([0.0] if own else list(np.array([0.8, 0.9, 1.0]) * top * (1 + 0.05 * j)))
            ln.append(len(lam[-1]))
            off.append(off[-1] + ln[-1])
    cat = lambda x: np.concatenate([np.asarray(a, dtype=np.float64) for a in x])
    return np.array(off, dtype=np.int64), cat(lam), cat(v), cat(res), np.array(ln, dtype=np.int32)


def _solve(off, lam, v, res, ln):
    d = [torch.from_numpy(x).cuda() for x in (off, lam, v, res, ln)]
    entries, cap = int(off[-1]), 64
    lib = l1line.load()
    ws = l1line.Workspace(int(lib.l1line_solution_path_workspace_bytes(M, entries)))
    st, ic, sl = (torch.zeros(cap, dtype=torch.float64, device="cuda") for _ in range(3))
    jh = torch.zeros(cap, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    rc = lib.l1line_solution_path_f64(
        M, *[x.data_ptr() for x in d], entries, st.data_ptr(), jh.data_ptr(), ic.data_ptr(),
        sl.data_ptr(), None, cnt.data_ptr(), cap, ctypes.c_void_p(ws.ptr), ws.nbytes,
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == l1line.OK
    c = min(int(cnt.item()), cap)
    return l1line.status(ws), st[:c].cpu(), jh[:c].cpu(), ic[:c].cpu(), sl[:c].cpu()


@pytest.mark.parametrize("top,lam_scale", [(4e307, 1.0), (1.0, 1.0), (1e-310, 1e-310),
                                           (3e-320, 1e-315)])
def test_objectives_at_the_range_ends(top, lam_scale):
    off, lam, v, res, ln = _paths(top, lam_scale)
    rc, st, jh, ic, sl = _solve(off, lam, v, res, ln)
    assert rc == l1line.OK and len(st) >= 1
    for q in (0.25 * lam_scale, 1.5 * lam_scale, 5.0 * lam_scale):
        z = [sum(float(res[off[p] + e]) + q * abs(float(v[off[p] + e]))
                 for p in range(j * M, j * M + M)
                 for e in [int(np.searchsorted(lam[off[p]:off[p] + ln[p]], q, side="right")) - 1])
             for j in range(M)]
        e = int(np.searchsorted(st.numpy(), q, side="right")) - 1
        got = float(ic[e]) + float(sl[e]) * q
        assert abs(got - min(z)) <= ((M + 8) * 2.0 ** -52 + 2e-12) * min(z) + (M + 8) * 2.0 ** -1074


@pytest.mark.parametrize("where", [0, 1, 2])
@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_residuals_that_are_not_finite(value, where):
    off, lam, v, res, ln = _paths(1.0, 1.0)
    res[int(off[1]) + where] = value
    assert _solve(off, lam, v, res, ln)[0] == l1line.ERR_NONFINITE

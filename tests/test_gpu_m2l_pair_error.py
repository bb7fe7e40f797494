"""Rounding of the per-pair M2L in symmetric storage, component by component,
against the D-tensors of the same offsets."""
import numpy as np
import pytest
import torch

from paper_1811_06332_gb300 import fmm as F

pytestmark = pytest.mark.gpu


def sym(p):
    return [(a, b, j - a - b) for j in range(p + 1) for a in range(j, -1, -1) for b in range(j - a, -1, -1)]


def exact(r, p):
    """All derivatives of 1/|r| in extended precision (Hermite-like auxiliary functions)."""
    r = r.astype(np.longdouble)
    ir2 = 1 / (r * r).sum(0)
    f = [np.sqrt(ir2)]
    for m in range(p):
        f.append(-(2 * m + 1) * ir2 * f[-1])
    rows = {(0, 0, 0): f}
    for k in sym(p)[1:]:
        d = next(i for i in range(3) if k[i])
        a = tuple(k[i] - (i == d) for i in range(3))
        v = [r[d] * rows[a][m + 1] for m in range(p - sum(k) + 1)]
        if a[d]:
            b = tuple(a[i] - (i == d) for i in range(3))
            v = [u + a[d] * rows[b][m + 1] for m, u in enumerate(v)]
        rows[k] = v
    return np.stack([rows[k][0] for k in sym(p)])


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("p", [2, 4, 6, 8, 10])
def test_monopoles_give_the_d_tensor(p, dtype):
    """M = (1, 0, ...): L_n = D_n.  The components that are summed have the D-tensor's own error; those that one step of
    the trace condition gives (nz = 2, 3 up to rank p - 3) the errors of two components: sqrt(2) times, as rms.  What is
    compared is the error of fmm_op_dtensor, the same recurrence."""
    o = np.array([v for v in np.ndindex(7, 7, 7)]) - 3
    r = np.ascontiguousarray(o[np.abs(o).max(1) >= 2].T.astype(np.float64))
    n, nc = r.shape[1], F.ncoef(p, F.BASIS_SYM)
    M = torch.zeros(nc, n, dtype=dtype, device="cuda")
    M[0] = 1.0
    L, D, rt = torch.empty_like(M), torch.empty_like(M), torch.from_numpy(r).cuda()
    prec = F.FP32 if dtype == torch.float32 else F.FP64
    F.fmm_op_m2l(p, F.BASIS_SYM, prec, M, rt, L)
    F.fmm_op_dtensor(p, prec, rt, D)
    torch.cuda.synchronize()
    ref = exact(r, p)
    scale = np.sqrt((ref * ref).mean(1))
    rms = [np.sqrt(((a.cpu().numpy() - ref) ** 2).mean(1)) for a in (L, D)]
    rank = np.array([sum(k) for k in sym(p)])
    eps = float(torch.finfo(dtype).eps)
    for j in range(p + 1):
        s = rank == j
        got, own = (np.sqrt((e[s] ** 2).sum() / (scale[s] ** 2).sum()) for e in rms)
        assert got <= 1.5 * own + eps / 8, (j, got, own)

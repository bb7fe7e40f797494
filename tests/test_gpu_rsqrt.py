"""The reciprocal square root of the FP64 near field, one pair at a time."""
import numpy as np
import pytest
import torch

from paper_1811_06332_gb300 import fmm as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("span", [0.5, 30.0, 500.0])
def test_within_one_ulp(span):
    """One unit charge at the origin, massless particles on the x axis: each potential is -1 / sqrt(fl(x^2)) alone.
    CUDA's rsqrt, which it replaces, is stated to be within 1 ulp."""
    n = 12_000
    rng = np.random.RandomState(int(span))
    x = 2.0 ** rng.uniform(-span, span, n)
    x[0] = 0.0
    q = np.zeros(n)
    q[0] = 1.0
    zero = np.zeros(n)
    plan = F.Plan(p=2, prec=F.FP64, adaptive=True, max_leaf=n, theta=0.0)
    plan.fmm_build_tree(*[torch.from_numpy(a).cuda() for a in (x, zero, zero, q)])
    out = torch.zeros(4, n, dtype=torch.float64, device="cuda")
    plan.fmm_p2p(*out)
    torch.cuda.synchronize()
    assert plan.stats()["leaves"] == 1
    plan.close()
    got = -out[0].cpu().numpy()[1:]
    ref = 1 / np.sqrt((x[1:] * x[1:]).astype(np.longdouble))
    ulp = np.spacing(ref.astype(np.float64)).astype(np.longdouble)
    assert np.max(np.abs(got - ref) / ulp) <= 1.0

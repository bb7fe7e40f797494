"""FP64 near field of massless and light particles at distances whose inverse
square leaves the FP64 range."""
import numpy as np
import pytest
import torch

from paper_1811_06332_gb300 import fmm as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg", [dict(depth=0), dict(depth=1), dict(adaptive=True, max_leaf=64, theta=0.0)])
@pytest.mark.parametrize("q1", [0.0, 1e-300])
def test_light_particle_very_near(cfg, q1):
    r = 2.0 ** -520   # 1 / r^2 = 2^1040 overflows, q1 / r^2 does not
    x = np.array([[0.0, r, 0.25, 0.3, 0.1], [0.0, 0.0, 0.25, 0.1, 0.3], [0.0, 0.0, 0.25, 0.2, 0.2]])
    q = np.array([1.0, q1, 0.5, 0.25, 0.0])
    plan = F.Plan(p=2, prec=F.FP64, **cfg)
    plan.fmm_build_tree(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (*x, q)])
    out = torch.zeros(4, 5, dtype=torch.float64, device="cuda")
    plan.fmm_p2p(*out)
    torch.cuda.synchronize()
    plan.close()
    got = out.cpu().numpy()
    for t in (0, 2, 3, 4):   # (target 1's field, 1 / r^2, is not representable)
        d = (x - x[:, t:t + 1]).astype(np.longdouble)
        rr = np.sqrt((d * d).sum(0))
        use = (rr > 0) & (q != 0.0)
        ir = 1 / rr[use]
        ref = np.array([-(q[use] * ir).sum(), *((q[use] * ir ** 3) * d[:, use]).sum(1)]).astype(float)
        # r^2 = 2^-1040 is subnormal with 34 bits; 1 / r follows it
        assert np.allclose(got[:, t], ref, rtol=2.0 ** -30, atol=0.0), (t, got[:, t], ref)

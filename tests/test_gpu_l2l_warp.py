"""L2L of the adaptive trees by a thread and by a warp per child: levels of both
sizes in one tree, against the oracle's field (FP64) and the FP64 plan (FP32)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1811_06332_gb300 import fmm as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("basis", [0, 1])
@pytest.mark.parametrize("p", range(0, 11))
def test_levels_of_both_forms(p, basis):
    n = 30_000   # leaves of at most 4: levels of 8 to 4096 cells, then of about 18,000
    rng = np.random.RandomState(p)
    x, q = rng.uniform(0, 1, (3, n)), rng.uniform(0.1, 1, n)
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (*x, q)]
    got = {}
    for prec in (F.FP64, F.FP32):
        plan = F.Plan(p=p, basis=basis, prec=prec, adaptive=True, max_leaf=4, theta=0.7)
        pot, acc = plan.evaluate(*t)
        torch.cuda.synchronize()
        got[prec] = torch.cat([pot[None], acc]).cpu().numpy()
        cells = plan.stats()["cells"]
        plan.close()
    assert cells > 3 * 4096
    s = np.arange(0, n, 997, dtype=np.int64)
    ref = oracle.fmm_adaptive(*x, q, 4, 0.7, p, basis, sample=s)
    ref = np.concatenate([ref[0][None], ref[1]])
    for rows in (slice(0, 1), slice(1, 4)):   # the stated tolerances of the forms
        assert np.linalg.norm(got[F.FP64][rows][:, s] - ref[rows]) <= 1e-12 * np.linalg.norm(ref[rows])
        assert np.linalg.norm(got[F.FP32][rows] - got[F.FP64][rows]) <= 5e-6 * np.linalg.norm(got[F.FP64][rows])

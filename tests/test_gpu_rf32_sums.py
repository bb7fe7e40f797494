"""Rounding of the uniform FP32 M2L on its small levels, whose lists are split
into shares and whose locals give most of the far potential."""
import numpy as np
import pytest
import torch

from paper_1811_06332_gb300 import fmm as F

pytestmark = pytest.mark.gpu


def far_potential(x, q, prec, depth):
    plan = F.Plan(p=0, prec=prec, depth=depth)
    t = [torch.from_numpy(a).cuda() for a in (*x, q)]
    out = torch.zeros(4, len(q), dtype=torch.float64, device="cuda")
    plan.fmm_build_tree(*t)
    plan.fmm_p2m(), plan.fmm_m2m(), plan.fmm_m2l(), plan.fmm_l2l()
    plan.fmm_l2p(*out)
    torch.cuda.synchronize()
    plan.close()
    return out[0].cpu().numpy()


@pytest.mark.parametrize("depth", [2, 3])
def test_potential_of_monopoles(depth):
    """p = 0: the far potential is the levels' sums of charge over distance.  Unit charges (exact multipoles and sums
    of sources): per orbit the D-tensor's and the product's rounding, each at most 2^-24 of the term, then the sum over
    the 56 shares rounded once, one rounding per level on the way down and one of the evaluation.  As rms: a rounding of
    a value uniform in its binade is below 0.42 * 2^-24; the orbits' average out."""
    rng = np.random.RandomState(depth)
    n = 40 * 8 ** depth
    x, q = rng.uniform(0, 1, (3, n)), np.ones(n)
    got, ref = far_potential(x, q, F.FP32, depth), far_potential(x, q, F.FP64, depth)
    rms = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    # terms: 2 roundings of each of the orbits over sqrt(7) (a share of the sum as uneven as the distances allow),
    # 1 of a level's sum, 1 per further level, 1 of the result
    assert rms <= 0.42 * 2.0 ** -24 * np.sqrt(2 / 7 + 1 + (depth - 2) + 1) * 1.5

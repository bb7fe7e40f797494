"""Storage of the mutual FP64 near field: held exactly where that form runs."""
import pytest
import torch

from paper_1811_06332_gb300 import fmm as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,depth,n,mutual", [(F.FP64, 3, 9000, 1), (F.FP64, 3, 8000, 0), (F.FP32, 3, 9000, 0),
                                                 (F.FP64, 7, 500_000, 0)])
def test_slots_follow_the_rule(prec, depth, n, mutual):
    x = torch.rand(4, n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    plan = F.Plan(p=0, prec=prec, depth=depth)
    plan.fmm_build_tree(*x)
    torch.cuda.synchronize()
    taken = free - torch.cuda.mem_get_info()[0]
    assert plan.stats()["p2p_mutual"] == mutual
    plan.close()
    if depth == 7:   # 27 n^2 / 8^7 = 3.2e6 pairs: 208 MB of slots beside about 110 MB of everything else
        assert taken < 416 * n

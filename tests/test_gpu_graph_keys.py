"""Captured steps against the buffers and arrays that they hold: a captured
graph must not outlive the plan's buffers, nor be replayed for other arrays."""
import numpy as np
import pytest
import torch

from paper_1811_06332_gb300 import fmm as F

pytestmark = pytest.mark.gpu


def arrays(n, seed):
    rng = np.random.RandomState(seed)
    return [torch.from_numpy(a).cuda() for a in (*rng.uniform(0, 1, (3, n)), rng.uniform(0.1, 1, n))]


def eager(X, **cfg):
    plan = F.Plan(**cfg)
    pot, acc = plan.evaluate(*X)
    torch.cuda.synchronize()
    plan.close()
    return torch.cat([pot[None], acc])


def equal(got, ref):
    # the same kernels on the same inputs, all sums in a fixed order
    return torch.equal(got, ref)


@pytest.mark.parametrize("cfg", [dict(p=4, basis=0, prec=F.FP64, depth=3), dict(p=6, basis=1, prec=F.FP32, depth=3),
                                 dict(p=4, basis=1, prec=F.GEMM_BF16X3, depth=5)])
def test_uniform_step_is_captured_again_after_another_size(cfg):
    n1, n2 = 9000, 4000
    A, B = arrays(n1, 1), arrays(n2, 2)
    out1 = torch.empty(4, n1, dtype=torch.float64, device="cuda")
    out2 = torch.empty(4, n2, dtype=torch.float64, device="cuda")
    plan, stream = F.Plan(use_graph=True, **cfg), torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    # an evaluation that allocates runs eagerly, the next of the same size captures
    for X, out, held in ((A, out1, 0), (A, out1, 1), (B, out2, 0), (A, out1, 0), (A, out1, 1), (A, out1, 1)):
        out.fill_(7.0)
        stream.wait_stream(torch.cuda.current_stream())
        plan.fmm_evaluate(*X, *out, stream=stream)
        stream.synchronize()
        assert plan.stats()["graph"] == held   # before anything is replayed into freed buffers
        assert equal(out, eager(X, **cfg))
    plan.close()


def test_host_entry_with_changing_sizes():
    """The staging buffers stay where they are when fewer particles follow."""
    cfg = dict(p=4, basis=0, prec=F.FP64, depth=3)
    plan, stream = F.Plan(use_graph=True, **cfg), torch.cuda.Stream()
    for n, held in ((9000, 0), (9000, 1), (4000, 0), (9000, 0), (9000, 1)):
        X = arrays(n, n)
        out = np.zeros((4, n))
        plan.fmm_evaluate_host(*[a.cpu().numpy() for a in X], *out, stream=stream)
        assert plan.stats()["graph"] == held
        assert np.array_equal(out, eager(X, **cfg).cpu().numpy())
    plan.close()

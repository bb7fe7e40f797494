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


def adaptive_outputs(plan, stream, X, out):
    for a in out:
        a.fill_(7.0)
    stream.wait_stream(torch.cuda.current_stream())
    plan.fmm_evaluate(*X, *out, stream=stream)
    stream.synchronize()


@pytest.mark.parametrize("swap", [0, 1, 2, 3])
def test_adaptive_replay_writes_the_arrays_it_is_given(swap):
    cfg = dict(p=4, basis=0, prec=F.FP32, adaptive=True, max_leaf=32, theta=0.6)
    X = arrays(5000, 3)
    plan, stream = F.Plan(use_graph=True, **cfg), torch.cuda.Stream()
    old = torch.empty(4, 5000, dtype=torch.float64, device="cuda")
    for _ in range(3):
        adaptive_outputs(plan, stream, X, old)
    assert plan.stats()["graph"] == 1
    ref, new = old.clone(), torch.empty_like(old)
    given = list(old)
    given[swap] = new[swap]   # one of the four is another array; the old ones stay allocated
    old[swap] = 3.0
    adaptive_outputs(plan, stream, X, given)
    assert torch.equal(torch.stack(given), ref)
    assert torch.all(old[swap] == 3.0)
    plan.close()


def test_learned_replay_follows_a_new_threshold():
    """The model's threshold shift (blob[6]) is held by value in the captured launches."""
    X = arrays(6000, 4)
    cfg = dict(p=6, basis=0, prec=F.FP32, adaptive=True, max_leaf=32, theta=0.6, learned_p=True, target_rel_err=1e-4)
    blob = np.zeros(F.MLP_NBLOB, dtype=np.float32)
    blob[:8] = [6332.0, 2.0, 12, 64, 9, 2.0, 0.0, 0.0]
    blob[20:32] = 1.0
    blob[-9:] = -np.arange(2, 11)   # the same log10 errors for every pair: order q gives 10^-q
    low = blob.copy()
    low[6] = 2.0                    # errors 100 times as large are accepted
    plan, stream = F.Plan(use_graph=True, **cfg), torch.cuda.Stream()
    out = torch.empty(4, 6000, dtype=torch.float64, device="cuda")
    got = []
    for b in (blob, low):
        plan.set_mlp(b)
        for _ in range(3):
            adaptive_outputs(plan, stream, X, out)
        got.append((out.clone(), plan.stats()["pairs_per_order"]))
    plan.close()
    for b, (res, per) in zip((blob, low), got):
        ep = F.Plan(**cfg)
        ep.set_mlp(b)
        pot, acc = ep.evaluate(*X)
        torch.cuda.synchronize()
        assert per == ep.stats()["pairs_per_order"]
        assert torch.equal(res, torch.cat([pot[None], acc]))
        ep.close()
    assert got[0][1] != got[1][1]

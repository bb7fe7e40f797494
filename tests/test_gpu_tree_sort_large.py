"""Lists of trees with more than 2^20 particles and pairs (the sorts' large
tiles), exactly: fields at FP64's rounding against the oracle's own lists."""
import numpy as np
import pytest
import torch

import oracle
from paper_1811_06332_gb300 import fmm as F

pytestmark = pytest.mark.gpu


def test_every_pair_once():
    """p = 2, so that the lists decide the result: a pair lost, doubled or given to another target changes a field by
    the pair's share of it, some 1e-6 and more with 2^20 particles; equal lists agree to 1e-12."""
    n = (1 << 20) + 1
    rng = np.random.RandomState(3)
    x, q = rng.normal(0, 1, (3, n)), rng.uniform(0.5, 1, n)
    s = np.sort(rng.choice(n, 300, replace=False)).astype(np.int64)
    pref, aref, st = oracle.fmm_adaptive(*x, q, 16, 0.6, 2, 0, sample=s)
    plan = F.Plan(p=2, prec=F.FP64, adaptive=True, max_leaf=16, theta=0.6)
    pot, acc = plan.evaluate(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (*x, q)])
    torch.cuda.synchronize()
    g = plan.stats()
    plan.close()
    assert st["p2p_pairs"] > 1 << 20 and st["m2l_pairs"] > 1 << 20
    assert (g["cells"], g["leaves"], g["m2l_pairs"], g["p2p_pairs"]) == (
        st["nodes"], st["leaves"], st["m2l_pairs"], st["p2p_pairs"])
    pot, acc = pot.cpu().numpy()[s], acc.cpu().numpy()[:, s]
    assert np.all(np.abs(pot - pref) <= 1e-12 * np.abs(pref))
    assert np.all(np.abs(acc - aref).max(0) <= 1e-10 * np.linalg.norm(aref, axis=0).mean())

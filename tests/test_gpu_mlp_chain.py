"""A long chain of training steps, whose kernels start before their
predecessors have ended, against the same steps launched one by one."""
import hashlib
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_1811_06332_gb300 import fmm as F
from paper_1811_06332_gb300 import order_model

pytestmark = pytest.mark.gpu

# 2432 samples a step: 304 blocks, two per SM; 256 samples: 32 blocks, the next step's beside them
CASES = [(2432 * 4, 2432, 75), (256 * 16, 256, 20)]


def train(n, batch, epochs):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    feat = torch.randn(n, 12, generator=g, device="cuda")
    lab = -4.0 + 2.0 * torch.randn(n, 9, generator=g, device="cuda")
    order = torch.randperm(n, generator=g, device="cuda").to(torch.int32)
    blob, losses = F.fmm_mlp_train(order_model.init_blob(5), feat, lab, order, epochs=epochs, batch=batch, lr=1e-3)
    assert np.all(np.isfinite(blob)) and losses[-1] < losses[0]
    return hashlib.sha256(blob.tobytes() + losses.tobytes()).hexdigest()


@pytest.fixture(scope="module")
def one_by_one():
    """The same trainings in a process whose launches each wait for their kernel."""
    env = dict(os.environ, CUDA_LAUNCH_BLOCKING="1", PYTHONPATH=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return r.stdout.split()


@pytest.mark.parametrize("k", range(len(CASES)))
def test_overlapping_steps_give_the_same_bits(one_by_one, k):
    # sums run in a fixed order, so a parameter or a partial sum read too early is the only way to differ
    for _ in range(3):
        assert train(*CASES[k]) == one_by_one[k]


if __name__ == "__main__":
    print(*[train(*c) for c in CASES])

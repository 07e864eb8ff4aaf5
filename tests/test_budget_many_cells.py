"""Budgets of sequences with more cells than a block has threads, so that the ranking of the fractional parts takes several turns:
80 layers of 8 KV heads by blocks of 256 and of 1024 threads, and numbers of cells just below and above one and two turns of
256.  Against the CPU oracle's one-at-a-time selection: whole numbers, equal."""
import numpy as np
import pytest
import torch

from harness import GpuPath
from workloads import Workload

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("layers,heads,batch", [(80, 8, 2), (80, 8, 1), (64, 4, 2), (63, 4, 4), (65, 4, 3), (64, 8, 3), (257, 2, 3)])
@pytest.mark.parametrize("ratio", [0.1, 0.5])
@pytest.mark.parametrize("alike", [False, True])
def test_budgets_of_many_cells(oracle_mod, layers, heads, batch, ratio, alike):
    """alike: groups of cells with the same scores, whose fractional parts are equal (the lower cell is taken first)."""
    n_visual = 67
    wl = Workload("cells", layers, heads, heads, 64, batch=batch, n_visual=n_visual, n_text=4, ratio=ratio, steps=1, window=2)
    rng = np.random.default_rng(layers * heads + batch)
    scores = np.exp(rng.standard_normal((layers, batch, heads, n_visual)) * rng.uniform(0.2, 1.5, (layers, batch, heads, 1)))
    scores = (scores / scores.sum(-1, keepdims=True)).astype(np.float32)
    if alike:
        scores[:] = scores[np.arange(layers) % 3][:, :, :1]
    strength, skewness = oracle_mod.moments(scores)
    want = oracle_mod.allocate_groups(strength, skewness, n_visual, ratio)
    gp = GpuPath(wl, device=DEV, per_kv_head=1)
    for _ in range(2):
        gp.budgets.fill_(-1)
        gp.budget(scores=torch.from_numpy(scores).to(DEV))
        assert gp.status() == 0
        assert np.array_equal(gp.budgets.cpu().numpy().reshape(want.shape), want)

"""Budgets and selection at the edges of their block sizes: many and few cells, token counts that fill the registers of a
block exactly and by one more, heavily duplicated scores (ties go to the lower index), a range of scores so wide that
the first histogram separates nothing, and scores that are all alike."""
import numpy as np
import pytest
import torch

from harness import GpuPath
from workloads import Workload

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("layers,batch", [(3, 2), (19, 16)])
@pytest.mark.parametrize("n_visual", [3, 255, 4096, 4097, 8192, 8193, 16385])
def test_budget_and_selection(oracle_mod, layers, batch, n_visual):
    wl = Workload("keep", layers, 1, 1, 64, batch=batch, n_visual=n_visual, n_text=2, ratio=0.23, steps=1, window=2)
    rng = np.random.default_rng(n_visual)
    scores = np.exp(rng.normal(size=(layers, batch, n_visual))).astype(np.float32)
    scores[0] = np.float32(rng.integers(0, 50, size=scores[0].shape) / 64.0)   # ties
    scores[1, 0, :] *= np.float32(1e-30)                                       # nearly all keys in one bin ...
    scores[1, 0, 0] = np.float32(1e30)                                         # ... of the first histogram
    scores[2, 0, :] = np.float32(0.125)                                        # all alike
    st, sk = oracle_mod.moments(scores)
    bud = oracle_mod.allocate(st, sk, n_visual, wl.ratio, 1)
    gp = GpuPath(wl, device=DEV)
    gp.set_full(*(torch.zeros((layers, batch, 1, n_visual + 2, 64), dtype=torch.bfloat16, device=DEV) for _ in range(2)))
    dev = torch.from_numpy(scores).to(DEV)
    for _ in range(2):   # the second call finds the tickets as the first left them
        gp.budget(scores=dev, mode=1)
        gp.compact(scores=dev)
    assert gp.status() == 0
    assert np.allclose(gp.strength.cpu().numpy(), st, rtol=1e-12, atol=0)
    assert np.allclose(gp.skew.cpu().numpy(), sk, rtol=1e-9, atol=1e-12)
    assert np.array_equal(gp.budgets.cpu().numpy(), bud)
    flat, k = scores.reshape(-1, n_visual), bud.reshape(-1)
    want = [np.sort(np.argsort(-flat[i], kind="stable")[:k[i]]) for i in range(len(k))]
    assert np.array_equal(gp.kept.cpu().numpy()[:int(k.sum())], np.concatenate(want))


@pytest.mark.parametrize("n_visual", [3, 40, 2916, 4097, 8193, 16385])
def test_a_sequence_alone_and_in_a_batch(n_visual):
    """Strength, skewness and budgets of a sequence do not depend, to the last bit, on how many sequences share the call (the
    kernel takes smaller blocks for many cells)."""
    layers, batch = 19, 24
    gen = torch.Generator(device=DEV).manual_seed(n_visual)
    scores = torch.exp(2 * torch.randn((layers, batch, n_visual), generator=gen, device=DEV))
    results = []
    for seqs in (list(range(batch)), [0], [5], [7, 23]):
        wl = Workload("alone", layers, 1, 1, 64, batch=len(seqs), n_visual=n_visual, n_text=2, ratio=0.23, steps=1, window=2)
        gp = GpuPath(wl, device=DEV)
        gp.budget(scores=scores[:, seqs].contiguous())
        assert gp.status() == 0
        got = (gp.strength.view(torch.int64), gp.skew.view(torch.int64), gp.budgets)
        if results:
            for a, b in zip(results, got):
                assert torch.equal(a[:, seqs], b)
        else:
            results = got

"""The cluster scoring kernel at the edges of its range: one tile, tile and block boundaries, the longest sequence it
takes and the first it does not, several units of 16 elite rows, and logits spread so far that the exponent reference
of a row has to move.  Against the CPU oracle, element by element, within the suite's 2e-3 (a logit of 100 in the
log2 domain, summed in fp32 over 128 exact products, is off by some 1e-4 at most)."""
import numpy as np
import pytest
import torch

from harness import GpuPath, gen_inputs, logical, oracle_dims, rel_elem_err, u16
from workloads import Workload

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n_visual,d,window,alpha,sharp,per_head", [
    (3, 128, 4, 0.9, 1.0, 0), (128, 64, 16, 0.9, 1.0, 0), (129, 128, 16, 0.9, 1.0, 1), (1025, 128, 16, 0.5, 1.0, 0),
    (2049, 64, 64, 0.3, 1.0, 0), (2500, 128, 16, 0.9, 6.0, 0), (3000, 64, 32, 0.2, 6.0, 1),
    (16384, 128, 16, 0.9, 1.0, 0), (16385, 128, 16, 0.9, 1.0, 0)])
def test_scores_at_the_edges(oracle_mod, n_visual, d, window, alpha, sharp, per_head):
    wl = Workload("edge", 2, 14, 2, d, batch=2, n_visual=n_visual, n_text=70, ratio=0.1, steps=1, window=window,
                  alpha=alpha)
    scale = sharp / d ** 0.5
    k, v, qw = gen_inputs(wl, "cpu")
    score = oracle_mod.score_groups if per_head else oracle_mod.score
    ref = score(oracle_dims(oracle_mod, wl), u16(logical(k)), u16(qw), scale, alpha)
    gp = GpuPath(wl, device=DEV, per_kv_head=per_head)
    gp.sh.scale = scale
    gp.set_full(logical(k.to(DEV)), logical(v.to(DEV)))
    for _ in range(2):   # the second call finds the workspace as the first left it
        gp.scores.fill_(float("nan"))
        gp.score(qw.to(DEV), alpha=alpha)
        assert gp.status() == 0
        assert np.array_equal(gp.mask.cpu().numpy().view(np.uint64), ref["elite_mask"])
        err = rel_elem_err(gp.scores.cpu().numpy(), ref["scores"])
        assert err <= 2e-3, err



@pytest.mark.parametrize("window", [4, 16, 31, 33, 64])
def test_ties_at_the_threshold(oracle_mod, window):
    """Candidates whose logits are equal in exact arithmetic (the query's channels are all alike and the keys are
    permutations of one another) and alpha = 1: all are elite, however an fp32 sum of their products would come out."""
    wl = Workload("ties", 1, 14, 2, 128, batch=2, n_visual=300, n_text=70, ratio=0.1, steps=1, window=window, alpha=1.0)
    k, v, qw = gen_inputs(wl, "cpu")
    gen = torch.Generator().manual_seed(1)
    row = k[0, 0, 0, 0].clone()
    for w in range(window):
        k[:, :, -1 - w] = row[torch.randperm(128, generator=gen)]
    qw[:, :, -1] = 0.37
    ref = oracle_mod.score(oracle_dims(oracle_mod, wl), u16(logical(k)), u16(qw), 0.1, 1.0)
    assert (ref["elite_mask"] == (1 << window) - 1).all()
    gp = GpuPath(wl, device=DEV)
    gp.sh.scale = 0.1
    gp.set_full(logical(k.to(DEV)), logical(v.to(DEV)))
    gp.score(qw.to(DEV), alpha=1.0)
    assert gp.status() == 0
    assert np.array_equal(gp.mask.cpu().numpy().view(np.uint64), ref["elite_mask"])


@pytest.mark.parametrize("n_visual,heads,d,window,sharp,per_head", [
    (3, (8, 2), 128, 8, 1.0, 0), (127, (14, 2), 64, 5, 1.0, 1), (128, (32, 2), 128, 64, 1.0, 0),
    (1000, (14, 2), 128, 64, 6.0, 0), (4097, (28, 4), 128, 16, 6.0, 1), (2500, (4, 4), 64, 128, 1.0, 0),
    (20000, (16, 1), 64, 9, 1.0, 0)])
def test_whole_window_at_the_edges(oracle_mod, n_visual, heads, d, window, sharp, per_head):
    """alpha = 0: one tile and fewer, query blocks that fill 128 rows and that do not, several of them, references that
    have to move, and a sequence cut into many pieces."""
    wl = Workload("edge0", 2, heads[0], heads[1], d, batch=2, n_visual=n_visual, n_text=130, ratio=0.1, steps=1,
                  window=window, alpha=0.0)
    scale = sharp / d ** 0.5
    k, v, qw = gen_inputs(wl, "cpu")
    score = oracle_mod.score_groups if per_head else oracle_mod.score
    ref = score(oracle_dims(oracle_mod, wl), u16(logical(k)), u16(qw), scale, 0.0)
    gp = GpuPath(wl, device=DEV, per_kv_head=per_head)
    gp.sh.scale = scale
    gp.set_full(logical(k.to(DEV)), logical(v.to(DEV)))
    for _ in range(2):
        gp.scores.fill_(float("nan"))
        gp.score(qw.to(DEV), alpha=0.0)
        assert gp.status() == 0
        assert np.array_equal(gp.mask.cpu().numpy().view(np.uint64), ref["elite_mask"])
        err = rel_elem_err(gp.scores.cpu().numpy(), ref["scores"])
        assert err <= 2e-3, err

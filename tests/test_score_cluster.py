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
    """alpha = 0: one tile and fewer, query blocks that fill 128 rows and that do not, several of them, logits up to six times
    as sharp (no reference moves for them: test_score_paths.py), and a sequence cut into many pieces."""
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


def masked_case(oracle_mod, edit, n_visual, window, alpha, d=128, heads=(14, 2)):
    """Scores of a case whose keys and window queries `edit` changes, and the oracle's.  Channel 0 of every query is positive
    and that of every key zero before: a key gets an extra logit by its channel 0."""
    wl = Workload("masked", 2, heads[0], heads[1], d, batch=1, n_visual=n_visual, n_text=70, ratio=0.1, steps=1,
                  window=window, alpha=alpha)
    k, v, qw = gen_inputs(wl, "cpu")
    qw[..., 0] = qw[..., 0].abs() + 0.125
    k[..., 0] = 0
    edit(k, qw)
    scale = 1 / d ** 0.5
    ref = oracle_mod.score(oracle_dims(oracle_mod, wl), u16(logical(k)), u16(qw), scale, alpha)
    gp = GpuPath(wl, device=DEV)
    gp.sh.scale = scale
    gp.set_full(logical(k.to(DEV)), logical(v.to(DEV)))
    gp.score(qw.to(DEV), alpha=alpha)
    assert gp.status() == 0
    assert np.array_equal(gp.mask.cpu().numpy().view(np.uint64), ref["elite_mask"])
    return gp.scores.cpu().numpy(), ref["scores"]


@pytest.mark.parametrize("value", [float("-inf"), -3.3e38])
@pytest.mark.parametrize("tokens", [(0, 1), (128, 131), (5, 290)])
@pytest.mark.parametrize("n_visual,window,alpha", [(300, 16, 0.9), (300, 2, 0.0), (3000, 16, 0.3)])
def test_masked_keys(oracle_mod, value, tokens, n_visual, window, alpha):
    """Keys that no query attends to (a channel of minus infinity, or so low that the logit overflows) score zero, also where
    such a key is the first that a thread meets, and the others score what they do without them."""
    def edit(k, qw):
        k[:, :, tokens[0]:tokens[1], :, 0] = value
    got, want = masked_case(oracle_mod, edit, n_visual, window, alpha)
    assert (want[..., tokens[0]:tokens[1]] == 0).all() and (want > 0).any()
    assert rel_elem_err(got, want) <= 2e-3


@pytest.mark.parametrize("low", [-1e30, -1e6, -1500.0])
@pytest.mark.parametrize("n_visual,window,alpha", [(300, 16, 0.9), (3000, 16, 0.9), (3000, 64, 0.2), (5000, 2, 0.0)])
def test_references_far_below(oracle_mod, low, n_visual, window, alpha):
    """The first key of every thread far below the others, so that its logit is no reference for them: the one that takes its
    place has to be exact beside it.  Logits up to 12 in magnitude otherwise: their rounding in 32 bits and that of a sum
    of 128 products is 2e-6 of a score; 2e-5 leaves room for the exponentials and the sums over keys."""
    def edit(k, qw):
        for tile in range(0, n_visual, 2048):
            k[:, :, tile:min(tile + 128, n_visual), :, 0] = low
    got, want = masked_case(oracle_mod, edit, n_visual, window, alpha)
    assert rel_elem_err(got, want) <= 2e-5


@pytest.mark.parametrize("n_visual", [300, 3000, 9000])
@pytest.mark.parametrize("window,alpha", [(16, 0.9), (2, 0.0)])
def test_scores_near_the_smallest(oracle_mod, n_visual, window, alpha):
    """Keys of 2^-104 of the largest weight, met by threads whose reference is 2^-127 of it: such a reference's own factor is
    below the smallest 32-bit number, the scores are not (5e-32), and a ranking of the tokens depends on them.  The oracle
    is compared above 1e-30 only, so the error of these scores is taken relative to themselves."""
    def edit(k, qw):
        k.zero_()
        qw.zero_()
        qw[..., :2] = 1.0
        put(k, slice(0, n_visual), -104.0)
        for tile in range(0, n_visual, 384):
            put(k, slice(tile, min(tile + 128, n_visual)), -127.0)
        put(k, 10, 0.0)
        put(k, slice(n_visual, None), -30.0)
    got, want = masked_case(oracle_mod, edit, n_visual, window, alpha)
    small = want > 2.0 ** -120
    assert small.sum() > want.size // 2
    assert (np.abs(got - want)[small] / want[small]).max() <= 2e-5


def put(k, tokens, x):
    """Keys whose logit is x in the log2 domain where the queries are one in two channels (the second for the bits) and zero
    in the others."""
    unit = np.log(2) * 128 ** 0.5
    hi = torch.tensor(x * unit).to(torch.bfloat16)
    k[:, :, tokens, :, 0] = hi
    k[:, :, tokens, :, 1] = (torch.tensor(x * unit) - hi.double()).to(torch.bfloat16)


@pytest.mark.parametrize("n_visual,loud", [(300, 10), (9000, 10), (300, 138), (3000, 266), (9000, 266)])
@pytest.mark.parametrize("below", [104, 124, 127, 135, 147])
def test_scores_far_below_a_key_of_the_same_warp(oracle_mod, n_visual, loud, below):
    """Keys of 2^-below of the largest weight, which a key of the same warp has, in its first tile (the reference from the
    start) or in a later one (the reference moves there), beside a few masked ones.  Subnormal scores are scores too: they are rounded to 2^-149 where
    an exponential is (weighted by the group's half), in the sum of a group and in the oracle, so two steps for two groups;
    beside that the 2e-5 of the other cases."""
    def edit(k, qw):
        k.zero_()
        qw.zero_()
        qw[..., :2] = 1.0
        put(k, slice(0, n_visual), -float(below))
        for tile in range(0, n_visual, 384):
            put(k, slice(tile, min(tile + 128, n_visual)), -127.0)
        put(k, loud, 0.0)
        put(k, slice(n_visual, None), -30.0)
        k[:, :, loud + 3:loud + 6, :, 0] = float("-inf")
    got, want = masked_case(oracle_mod, edit, n_visual, 2, 0.0)
    assert ((want > 0).sum(-1) == n_visual - 3).all()
    assert (np.abs(got.astype(np.float64) - want) <= 2 * 2.0 ** -149 + 2e-5 * want.astype(np.float64)).all()


@pytest.mark.parametrize("heads,d,window,alpha,n_visual", [
    ((8, 4), 64, 16, 0.9, 32), ((8, 4), 64, 16, 0.9, 33), ((8, 4), 64, 16, 0.5, 96), ((8, 4), 64, 16, 0.5, 97),
    ((4, 4), 128, 64, 0.9, 3), ((4, 4), 128, 70, 0.9, 3), ((32, 4), 64, 16, 0.3, 48), ((32, 4), 64, 16, 0.3, 49),
    ((8, 4), 64, 16, 0.9, 31)])
@pytest.mark.parametrize("batch,per_head", [(8, 0), (7, 0), (8, 1)])
def test_many_groups_of_hardly_a_tile(oracle_mod, heads, d, window, alpha, n_visual, batch, per_head):
    """Both sides of the lines between the cluster kernel and the older ones where a call covers many groups of few keys (896
    groups on 148 SMs are enough, 784 are not).  Logits of a few units, some hundred terms to a sum: 2e-5."""
    wl = Workload("hardly", 28, heads[0], heads[1], d, batch=batch, n_visual=n_visual, n_text=80, ratio=0.1, steps=1,
                  window=window, alpha=alpha)
    k, v, qw = gen_inputs(wl, "cpu")
    score = oracle_mod.score_groups if per_head else oracle_mod.score
    ref = score(oracle_dims(oracle_mod, wl), u16(logical(k)), u16(qw), wl.scale, alpha)
    gp = GpuPath(wl, device=DEV, per_kv_head=per_head)
    gp.set_full(logical(k.to(DEV)), logical(v.to(DEV)))
    gp.score(qw.to(DEV), alpha=alpha)
    assert gp.status() == 0
    assert np.array_equal(gp.mask.cpu().numpy().view(np.uint64), ref["elite_mask"])
    assert rel_elem_err(gp.scores.cpu().numpy(), ref["scores"]) <= 2e-5

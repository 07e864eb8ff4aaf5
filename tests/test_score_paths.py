"""Scoring calls that the usual shapes do not reach: references that have to move in the whole-window passes, candidates at
the threshold for alpha below one, and the older kernels, which take long sequences, caches that no tensor map describes
and windows too wide for the cluster kernel.  Against the CPU oracle.

Bound: logits are 32-bit sums of exact products, rounded at 2^-24 of their magnitude a few times, so a score is off by
some 2^-22 times its largest logit in the log2 domain: 3e-6 at 12, 4e-5 at 170."""
import numpy as np
import pytest
import torch

from harness import GpuPath, gen_inputs, logical, oracle_dims, rel_elem_err, u16
from workloads import Workload

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def workload(layers, heads, d, batch, n_visual, window, alpha, n_text=None):
    return Workload("paths", layers, heads[0], heads[1], d, batch=batch, n_visual=n_visual, n_text=n_text or window + 30,
                    ratio=0.1, steps=1, window=window, alpha=alpha)


def compare(oracle_mod, wl, k, v, qw, bound, per_head=0, full=None, scale=None):
    """`full`: the device view of the keys and values, if it is not the plain one."""
    scale = scale or wl.scale
    score = oracle_mod.score_groups if per_head else oracle_mod.score
    ref = score(oracle_dims(oracle_mod, wl), u16(logical(k)), u16(qw), scale, wl.alpha)
    gp = GpuPath(wl, device=DEV, per_kv_head=per_head)
    gp.sh.scale = scale
    gp.set_full(*(full or (logical(k.to(DEV)), logical(v.to(DEV)))))
    for _ in range(2):   # the second call finds the workspace as the first left it
        gp.scores.fill_(float("nan"))
        gp.score(qw.to(DEV), alpha=wl.alpha)
        assert gp.status() == 0
        assert np.array_equal(gp.mask.cpu().numpy().view(np.uint64), ref["elite_mask"])
        err = rel_elem_err(gp.scores.cpu().numpy(), ref["scores"])
        assert err <= bound, err


@pytest.mark.parametrize("n_visual,later", [(128, 64), (300, 200), (90000, 5 * 128 + 70), (90000, 13 * 128 + 1)])
@pytest.mark.parametrize("heads,window", [((14, 2), 16), ((16, 1), 9)])
def test_whole_window_references_that_move(oracle_mod, heads, window, n_visual, later):
    """alpha = 0, pass one: a row's reference is the largest logit of the first 32 keys its thread meets and moves when the
    sum of 32 keys passes 2^60.  Quiet keys first, then single keys 80 above them in the log2 domain: later in the same
    tile, in the next, and in a later tile of the same epilogue set, which a block meets in pieces of more than four."""
    wl = workload(1, heads, 64, 1, n_visual, window, 0.0)
    k, v, qw = gen_inputs(wl, "cpu")
    k, qw = k * 0.25, qw * 0.25
    qw[..., 0], k[..., 0] = 2.0, 0.0
    scale = 0.125
    loud = 80 * np.log(2) / (2.0 * scale)
    k[:, :, later:n_visual:2531, :, 0] = loud
    # the condition the test is there for, on the logits themselves: quiet in the thread's first 32 keys, above 60 later
    log2 = torch.einsum("wd,nd->wn", qw[0, 0, :, 0].float(), k[0, 0, :n_visual, 0].float()) * (scale / np.log(2))
    first = log2[:, later // 32 * 32 - 32:later // 32 * 32].amax(1) if later >= 32 else log2[:, :32].amax(1)
    assert (log2[:, later] - first > 62).all() and (log2[:, :32].amax(1) < 12).all()
    compare(oracle_mod, wl, k, v, qw, 5e-5, scale=scale)


@pytest.mark.parametrize("window", [16, 31, 64])
@pytest.mark.parametrize("alpha", [0.9, 0.5, 0.2])
def test_candidates_at_the_threshold(oracle_mod, window, alpha):
    """Candidates whose logits lie within a few units in the last place of the threshold, on both sides, beside others far from
    it: the fp32 decision cannot settle them and the fp64 one has to agree with the oracle's bit for bit.  Scales next to
    one another move them across the line."""
    wl = workload(1, (14, 2), 128, 2, 300, window, alpha)
    k, v, qw = gen_inputs(wl, "cpu")
    gen = torch.Generator().manual_seed(7)
    last = torch.randn(128, generator=gen).to(torch.bfloat16)
    qw[:, :, -1] = last
    best = torch.randn(128, generator=gen).to(torch.bfloat16)
    best[:32] = last[:32]
    top = float(best.double() @ last.double())
    assert top > 8
    wanted = np.log(alpha) / 0.09   # below the best logit, before the scale
    for w in range(window):
        row = best.clone()
        if w % 3 == 1:     # far below
            row = -best
        elif w % 3 == 2:   # channel after channel closer to the threshold, then its last channels in small steps
            row = torch.randn(128, generator=gen).to(torch.bfloat16)
            for c in range(96, 128):
                left = top + wanted - (float(row.double() @ last.double()) - float(row[c].double() * last[c].double()))
                row[c] = torch.tensor(left / float(last[c])).to(torch.bfloat16) if abs(float(last[c])) > 0.05 else row[c]
        k[:, :, -window + w] = row
    sides = set()
    for i in range(-6, 7):
        scale = float(np.float32(0.09) * np.float32(1 + i * 2e-7))
        dm = oracle_dims(oracle_mod, wl)
        ref = oracle_mod.score(dm, u16(logical(k)), u16(qw), scale, alpha)
        gp = GpuPath(wl, device=DEV)
        gp.sh.scale = scale
        gp.set_full(logical(k.to(DEV)), logical(v.to(DEV)))
        gp.score(qw.to(DEV), alpha=alpha)
        assert gp.status() == 0
        assert np.array_equal(gp.mask.cpu().numpy().view(np.uint64), ref["elite_mask"])
        sides.add(int(ref["elite_mask"].reshape(-1)[0]))
    close = [abs(float(k[0, 0, -window + w, 0].double() @ last.double()) - top - wanted) for w in range(2, window, 3)]
    size = max(float((k[0, 0, -window + w, 0].double() * last.double()).abs().sum()) for w in range(window))
    assert min(close) < 9e-6 * size, "no candidate is as close as the fp32 decision's slack"


def logit_sum_fp32(q, k):
    """The kernel's fp32 dot product: even and odd channels in element order, then one addition."""
    sums = [np.float32(0), np.float32(0)]
    for c, x in enumerate((q.double() * k.double()).tolist()):
        sums[c & 1] = np.float32(float(sums[c & 1]) + x)
    return np.float32(sums[0] + sums[1])


@pytest.mark.parametrize("window", [8, 32, 33, 128])
def test_candidates_that_cancel_at_the_threshold(oracle_mod, window):
    """Candidates whose products are large and cancel, within some 1e-4 of the threshold on both sides: their fp32 sums are off by
    more than that and decide several of them wrongly, the sum of the products' magnitudes (the slack, taken by shuffles up
    to 32 candidates and by an atomic maximum beyond) has to send them to the fp64 sums."""
    alpha, scale = 0.5, 0.09
    wl = workload(1, (14, 2), 128, 1, 300, window, alpha, n_text=window + 3)
    k, v, qw = gen_inputs(wl, "cpu")
    gen = torch.Generator().manual_seed(window)
    last = torch.randn(128, generator=gen).to(torch.bfloat16)
    last[64:] = last[:64]
    last[127], last[63] = 2.0 ** -5, 2.0 ** -14   # two channels to aim with, the others cancel
    qw[:, :, -1] = last
    q = last.double()
    wanted = np.log(alpha) / scale   # below the best candidate's logit, which is zero
    exact, rough = [], []
    for w in range(window):
        row = torch.zeros(128, dtype=torch.bfloat16)
        if w:
            row[:63] = (300 * torch.randn(63, generator=gen)).to(torch.bfloat16)
            row[64:127] = -row[:63]
            aim = wanted + (w - window / 2) * 2e-4 / window
            for c in (127, 63):
                row[c] = torch.tensor((aim - float(row.double() @ q)) / float(q[c])).to(torch.bfloat16)
            exact.append(float(row.double() @ q) - wanted)
            rough.append(float(logit_sum_fp32(last, row)) - wanted)
            assert abs(exact[-1]) < 9e-6 * float((row.double() * q).abs().sum())
        k[:, :, -window + w] = row
    assert any((a > 0) != (b > 0) for a, b in zip(exact, rough)), "fp32 sums decide as the exact ones do"
    assert min(exact) < 0 < max(exact)
    dm = oracle_dims(oracle_mod, wl)
    ref = oracle_mod.score(dm, u16(logical(k)), u16(qw), scale, alpha)
    gp = GpuPath(wl, device=DEV)
    gp.sh.scale = scale
    gp.set_full(logical(k.to(DEV)), logical(v.to(DEV)))
    gp.score(qw.to(DEV), alpha=alpha)
    assert gp.status() == 0
    assert np.array_equal(gp.mask.cpu().numpy().view(np.uint64), ref["elite_mask"])


@pytest.mark.parametrize("heads,d,window,alpha,n_visual,per_head", [
    ((14, 2), 64, 16, 0.9, 16385, 0), ((14, 2), 64, 64, 0.2, 17000, 0), ((16, 8), 128, 64, 0.1, 16500, 1),
    ((8, 8), 64, 32, 0.9, 40000, 1), ((16, 1), 128, 16, 0.5, 33000, 0), ((2, 1), 128, 9, 0.0, 20000, 0)])
def test_longer_than_a_cluster_holds(oracle_mod, heads, d, window, alpha, n_visual, per_head):
    """The one-pass kernel: both head dims, per-KV-head scores, more than the 16 elite rows whose logits it keeps, and every
    window query of a small group."""
    wl = workload(1, heads, d, 1, n_visual, window, alpha)
    k, v, qw = gen_inputs(wl, "cpu")
    compare(oracle_mod, wl, k, v, qw, 2e-5, per_head)


@pytest.mark.parametrize("alpha,window", [(0.9, 16), (0.3, 64), (0.0, 16), (0.0, 2)])
@pytest.mark.parametrize("shared", ["batch", "layer"])
@pytest.mark.parametrize("per_head", [0, 1])
def test_one_copy_of_the_keys_shared(oracle_mod, alpha, window, shared, per_head):
    """A stride of zero, one prompt's keys for all sequences or layers: no tensor map describes that, so neither the cluster
    kernel nor the whole-window passes take the call."""
    wl = workload(3, (14, 2), 128, 3, 700, window, alpha)
    k, v, qw = gen_inputs(wl, "cpu")
    axis = 1 if shared == "batch" else 0
    k, v = (t.narrow(axis, 0, 1).expand(t.shape) for t in (k, v))
    full = tuple(logical(t.narrow(axis, 0, 1).to(DEV)).expand(logical(k).shape) for t in (k, v))
    assert full[0].stride(axis) == 0
    compare(oracle_mod, wl, k.contiguous(), v.contiguous(), qw, 2e-5, per_head, full)


@pytest.mark.parametrize("heads,d,window", [((16, 2), 128, 128), ((16, 1), 128, 128), ((14, 2), 128, 128), ((16, 1), 64, 128)])
@pytest.mark.parametrize("alpha", [0.9, 0.2])
def test_windows_wide_for_the_cluster(oracle_mod, heads, d, window, alpha):
    """128 candidates of 128 channels and the last queries of eight heads leave no room for two ring stages (the older kernels
    take these calls), of seven heads or 64 channels they do."""
    wl = workload(1, heads, d, 2, 900, window, alpha)
    k, v, qw = gen_inputs(wl, "cpu")
    compare(oracle_mod, wl, k, v, qw, 2e-5)


@pytest.mark.parametrize("heads,window", [((14, 2), 5), ((14, 2), 9), ((16, 1), 19), ((14, 2), 16), ((3, 1), 43)])
def test_whole_window_masked_keys(oracle_mod, heads, window):
    """Keys of minus infinity in the whole-window passes score zero, also where the window rows of a KV group do not fill the
    last sixteen columns of a query block (35, 63, 129 in two blocks of up to 66) or do (304 in three, 112)."""
    wl = workload(2, heads, 128, 1, 700, window, 0.0)
    k, v, qw = gen_inputs(wl, "cpu")
    qw[..., 0], k[..., 0] = qw[..., 0].abs() + 0.125, 0.0
    k[:, :, 3:6, :, 0] = float("-inf")
    k[:, :, 128:450, :, 0] = float("-inf")
    compare(oracle_mod, wl, k, v, qw, 2e-5)

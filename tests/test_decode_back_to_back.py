"""Decode steps as a decoder issues them: one behind the other on a stream, nothing between them that waits, so that a
launch starts while the one before it ends, reads lengths that are being raised and plans over units that come to be.
Every step's output, the lengths and the cache against a softmax in 64 bits over the rows that the step has to see.

Bound: probabilities enter the second product as two 16-bit parts (2^-17 of a value), logits below 16 are rounded in 32
bits (2^-20 of a probability), sums of some hundred terms add as much again; 1e-4 of a row's largest value leaves room for
all of it, and a row too many, too few or in the wrong place is off by a hundredth at least."""
import numpy as np
import pytest
import torch

import paper_2503_23956_b200 as ac
from harness import rel_row_err

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def run_steps(layers, hq, hkv, d, lens, steps, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    normal = lambda *shape: torch.randn(shape, generator=gen, device=DEV).to(torch.bfloat16)
    lens = torch.tensor(lens, dtype=torch.int64, device=DEV)
    room = lens + steps
    offsets = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(room, 0)])
    rows = int(offsets[-1])
    k, v = normal(rows, hkv, d), normal(rows, hkv, d)
    q, kn, vn = normal(steps, layers, 1, hq, d), normal(steps, layers, 1, hkv, d), normal(steps, layers, 1, hkv, d)
    # the rows as the last step sees them, padded to the longest region
    width = int(room.max())
    at = (offsets[:-1, None] + torch.arange(width, device=DEV)).clamp(max=rows - 1)
    own = torch.arange(width, device=DEV) < room[:, None]
    want_k, want_v = k.clone(), v.clone()
    for i in range(steps):
        want_k[offsets[:-1] + lens + i], want_v[offsets[:-1] + lens + i] = kn[i, :, 0], vn[i, :, 0]
    kk, vv = (t[at].double().repeat_interleave(hq // hkv, dim=2) for t in (want_k, want_v))
    logits = torch.einsum("srhd,rnhd->srhn", q[:, :, 0].double(), kk) / d ** 0.5
    seen = torch.arange(width, device=DEV) < (lens + torch.arange(1, steps + 1, device=DEV)[:, None])[..., None]
    logits.masked_fill_(~(seen & own)[:, :, None], float("-inf"))
    want = torch.einsum("srhn,rnhd->srhd", torch.softmax(logits, dim=-1), vv)

    sh = ac.shape(layers, 1, hq, hkv, d, 8, 4, 2, steps)
    ws = torch.empty(ac.aircache_workspace_bytes(sh), dtype=torch.uint8, device=DEV)
    ac.aircache_reset_status(ws)
    ln = lens.to(torch.int32)
    cache = ac.ragged_view(k, v, offsets, ln, rows)
    out = torch.empty((steps, layers, 1, hq, d), device=DEV)
    torch.cuda.synchronize()
    for i in range(steps):
        ac.aircache_decode_step(sh, cache, q[i], kn[i], vn[i], i, out[i], ws)
    assert ac.aircache_check_status(ws, check=False) == 0
    assert torch.equal(ln, (lens + steps).to(torch.int32))
    assert torch.equal(k.view(torch.int16), want_k.view(torch.int16))
    assert torch.equal(v.view(torch.int16), want_v.view(torch.int16))
    for i in range(steps):
        err = rel_row_err(out[i, :, 0].cpu().numpy(), want[i].cpu().numpy())
        assert err <= 1e-4, (i, err)


@pytest.mark.parametrize("layers,hq,hkv,d", [
    (4, 14, 2, 128), (16, 8, 8, 64), (28, 32, 2, 128),   # a CTA per (region, KV head) and more CTAs than items
    (60, 7, 1, 64), (64, 28, 4, 128)])                   # by region, planned in registers
def test_steps_planned_in_registers(layers, hq, hkv, d):
    """The CTA that ends last raises the lengths, while warps of other CTAs may still be about to read them."""
    rng = np.random.default_rng(layers)
    run_steps(layers, hq, hkv, d, rng.integers(1, 200, layers).tolist(), 24, layers)


@pytest.mark.parametrize("layers,hq,hkv,d,first,steps", [
    (4, 14, 2, 128, 120, 150),    # units of 128 rows: the kept plan is replaced on the way to 129 rows and to 257
    (28, 28, 4, 64, 250, 20),     # whole items and pieces change places
    (60, 16, 8, 128, 9, 40)])     # by region, units of 16 rows
def test_steps_over_the_ends_of_units(layers, hq, hkv, d, first, steps):
    """Where a region's unit count changes, the plan kept in the workspace fits no more: every block makes a new one and
    keeps that, while its warps still compare the old one."""
    run_steps(layers, hq, hkv, d, [first + i % 11 for i in range(layers)], steps, layers)


@pytest.mark.parametrize("layers,hq,hkv,d", [
    (80, 28, 4, 128), (112, 8, 8, 64), (90, 64, 8, 128), (200, 3, 1, 128), (70, 32, 2, 64)])
def test_steps_over_shared_tables(layers, hq, hkv, d):
    """More regions than the register plan takes: the tables are built ahead of the dependency wait from lengths that the
    step before is raising, and built again where they turn out stale (some region opens a unit at every step); the
    consumers read a region's rows as they come to it and draw the ticket at the end.  With eight KV heads a warp has a
    head to itself and meets no other on its way."""
    rng = np.random.default_rng(layers)
    run_steps(layers, hq, hkv, d, rng.integers(0, 140, layers).tolist(), 40, layers)


@pytest.mark.parametrize("most", [25, 45])
@pytest.mark.parametrize("layers,hq,hkv,d", [(460, 7, 1, 128), (450, 8, 2, 64), (460, 4, 1, 64), (440, 7, 1, 128)])
def test_steps_over_many_short_regions(layers, hq, hkv, d, most):
    """More than three regions to a block, of few rows: there the tables are built behind the dependency wait only, unless
    two blocks share an SM or the buffers hold five eighths of a unit (40 rows here) a region: both sides of each line."""
    rng = np.random.default_rng(layers)
    run_steps(layers, hq, hkv, d, rng.integers(most - 12, most + 12, layers).tolist(), 7, layers)


@pytest.mark.parametrize("layers,batch,hq,hkv,d", [(28, 4, 28, 4, 128), (30, 3, 8, 8, 64), (40, 2, 4, 1, 128)])
def test_new_layouts_back_to_back(layers, batch, hq, hkv, d):
    """Scores, budgets, compaction and a decode call in a row, again and again into the same cache, without a wait: the
    decode call's tables are read early and then belong to the layout before.  Bit for bit what the same calls give with
    a wait behind each."""
    gen = torch.Generator(device=DEV).manual_seed(batch)
    normal = lambda *shape: torch.randn(shape, generator=gen, device=DEV).to(torch.bfloat16)
    nv, nt, window, rounds = 300, 20, 8, 6
    from paper_2503_23956_b200.session import Session
    s = Session(ac.shape(layers, batch, hq, hkv, d, nv, nt, window), 0.2, 0.9, DEV)
    k, v = (normal(layers, batch, hkv, nv + nt, d) for _ in range(2))
    s.set_full(k, v)
    qw = normal(rounds, layers, batch, window, hq, d)
    qw *= torch.linspace(0.3, 3, layers, device=DEV).to(torch.bfloat16)[:, None, None, None, None]
    q = normal(layers, batch, hq, d)
    results = []
    for wait in (True, False):
        s.k_c.zero_(), s.v_c.zero_(), s.lens.zero_(), s.offsets.zero_()
        out = torch.empty((rounds,) + tuple(s.out.shape), device=DEV)
        kept = torch.empty((rounds, s.kept_n), dtype=torch.int32, device=DEV)
        torch.cuda.synchronize()
        for i in range(rounds):
            for call in (lambda: s.score(qw[i]), s.budget, s.compact, lambda: s.decode(q, out[i])):
                call()
                if wait:
                    torch.cuda.synchronize()
            kept[i].copy_(s.kept)
        assert s.status() == 0
        results.append((out, kept, s.k_c.clone(), s.lens.clone()))
    assert not torch.equal(results[0][1][0], results[0][1][1])   # the layouts do differ
    for a, b in zip(*results):
        assert torch.equal(a, b)

"""Copying of text rows beside the selection: selection by fewer blocks than regions (blocks of 256 and 512 threads that take
two regions one after the other, and as many regions as blocks), text rows by blocks of their own and by those of the kept rows,
and short rows side by side in a warp.  Lists and rows against a library sort and plain indexing (whole numbers and copies:
equal)."""
import pytest
import torch

from harness import GpuPath
from workloads import Workload

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def check_compaction(layers, batch, heads, d, n_visual, n_text, ratio, per_head=0):
    wl = Workload("text", layers, heads, heads, d, batch=batch, n_visual=n_visual, n_text=n_text, ratio=ratio, steps=1, window=2)
    gen = torch.Generator(device=DEV).manual_seed(n_visual)
    full = [torch.empty((layers, batch, heads, n_visual + n_text, d), dtype=torch.bfloat16, device=DEV).normal_(generator=gen)
            for _ in range(2)]
    gp = GpuPath(wl, device=DEV, per_kv_head=per_head)
    scores = torch.exp(torch.randn(tuple(gp.scores.shape), generator=gen, device=DEV))
    gp.set_full(*full)
    gp.budget(scores=scores)
    for _ in range(2):
        gp.kept.fill_(-1)
        gp.k_c.fill_(float("nan"))
        gp.v_c.fill_(float("nan"))
        gp.compact(scores=scores)
    assert gp.status() == 0
    order = torch.sort(scores.view(-1, n_visual), dim=1, descending=True, stable=True).indices
    budgets, offsets = gp.budgets.view(-1).tolist(), gp.offsets.tolist()
    cells = heads if per_head else 1
    at = 0
    for r, k in enumerate(budgets):
        kept = torch.sort(order[r, :k]).values
        assert torch.equal(gp.kept[at:at + k].long(), kept)
        at += k
        rows = torch.cat([kept, torch.arange(n_visual, n_visual + n_text, device=DEV)])
        l, b, g = r // cells // batch, r // cells % batch, r % cells
        for have, src in ((gp.k_c, full[0]), (gp.v_c, full[1])):
            want = src[l, b, g:g + 1 if per_head else heads][:, rows].transpose(0, 1)
            assert torch.equal(have[offsets[r]:offsets[r] + k + n_text].view(-1), want.reshape(-1))


@pytest.mark.parametrize("layers,batch,d,n_visual,n_text", [
    (19, 16, 128, 300, 60),     # 304 regions, 256 threads
    (37, 8, 128, 4096, 50),     # 296 regions
    (37, 16, 128, 2000, 40),    # 592 regions by 296 blocks: exactly two each
    (30, 10, 128, 4097, 100),   # 300 regions by 148 blocks of 512 threads
    (30, 5, 64, 4097, 260),     # 150 regions, 512 threads
    (37, 4, 64, 4500, 140)])    # 148 regions: a block of 1024 threads each
def test_compaction_with_many_text_rows(layers, batch, d, n_visual, n_text):
    check_compaction(layers, batch, 8, d, n_visual, n_text, 0.07)


@pytest.mark.parametrize("layers,batch,heads,d,n_visual,n_text,ratio,per_head", [
    (28, 2, 4, 128, 1000, 16, 0.1, 0),     # shared: one kept block more on some SMs
    (28, 2, 4, 128, 1000, 70, 0.1, 0),     # apart: more text blocks than free SMs
    (28, 8, 4, 128, 300, 32, 0.1, 0),      # shared: either kind starts beside the selection, not both
    (28, 8, 4, 128, 300, 3, 0.5, 0),       # many kept, few text blocks
    (28, 8, 4, 128, 40, 64, 0.05, 0),      # few kept, many text blocks
    (37, 4, 4, 128, 50, 3, 0.1, 0),        # no SM is free beside the selection
    (3, 1, 4, 64, 77, 2, 0.02, 0),         # 32 vectors of a row: one row a warp
    (5, 2, 1, 64, 97, 5, 0.2, 0),          # 8: four rows abreast
    (7, 3, 2, 64, 333, 21, 0.3, 0),        # 16: two
    (5, 2, 8, 64, 97, 5, 0.2, 1),          # the same with budgets per KV head
    (9, 5, 4, 128, 301, 33, 0.1, 1),
    (4, 1, 2, 64, 5, 2, 1.0, 0)])
def test_text_and_kept_rows_in_one_block_or_two(layers, batch, heads, d, n_visual, n_text, ratio, per_head):
    check_compaction(layers, batch, heads, d, n_visual, n_text, ratio, per_head)

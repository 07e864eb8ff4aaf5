"""The fused decode step where the appended token falls on an edge: first or last row of a 16-row block or of a unit, the
row that opens a new unit, the only row of an empty region; in every cut of the work (by KV head, by region, by the shared
tables).  Against an fp32 softmax over the same rows, within the suite's 2e-3 of the row's largest value."""
import pytest
import torch

import paper_2503_23956_b200 as ac
from harness import rel_row_err

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
EDGES = [0, 1, 15, 16, 17, 31, 32, 63, 64, 65, 127, 128, 129, 255, 256, 300]


@pytest.mark.parametrize("layers,hq,hkv,d", [
    (4, 14, 2, 128), (16, 8, 4, 64), (16, 8, 8, 128), (16, 32, 2, 128),      # by KV head / by region, small and wide groups
    (80, 14, 2, 64), (80, 28, 4, 128), (112, 8, 8, 64), (200, 3, 1, 128)])   # more regions than the register plan takes
@pytest.mark.parametrize("empty", [False, True])
def test_token_at_an_edge(layers, hq, hkv, d, empty):
    gen = torch.Generator().manual_seed(layers)
    edges = EDGES if empty else EDGES[1:]
    lens = torch.tensor([edges[i % len(edges)] for i in range(layers)])
    slack = 3
    offsets = torch.cat([torch.zeros(1, dtype=torch.int64), torch.cumsum(lens + slack, 0)])
    rows = int(offsets[-1])
    k, v = (torch.randn((rows, hkv, d), generator=gen).to(torch.bfloat16) for _ in range(2))
    for r in range(layers):   # what lies in the slack must not matter
        k[offsets[r] + lens[r]:offsets[r + 1]] = float("nan")
        v[offsets[r] + lens[r]:offsets[r + 1]] = float("nan")
    sh = ac.shape(layers, 1, hq, hkv, d, 8, 4, 2, slack)
    ws = torch.empty(ac.aircache_workspace_bytes(sh), dtype=torch.uint8, device=DEV)
    ac.aircache_reset_status(ws)
    kc, vc, off, ln = k.to(DEV), v.to(DEV), offsets.to(DEV), lens.to(torch.int32).to(DEV)
    cache = ac.ragged_view(kc, vc, off, ln, rows)
    out = torch.empty((layers, 1, hq, d), device=DEV)
    for step in range(2):
        q = torch.randn((layers, 1, hq, d), generator=gen).to(torch.bfloat16)
        kn, vn = (torch.randn((layers, 1, hkv, d), generator=gen).to(torch.bfloat16) for _ in range(2))
        ac.aircache_decode_step(sh, cache, q.to(DEV), kn.to(DEV), vn.to(DEV), step, out, ws)
        assert ac.aircache_check_status(ws, check=False) == 0
        want = torch.empty((layers, hq, d))
        for r in range(layers):
            n = int(lens[r]) + step
            k[offsets[r] + n], v[offsets[r] + n] = kn[r, 0], vn[r, 0]
            kr, vr = (t[offsets[r]:offsets[r] + n + 1].float().repeat_interleave(hq // hkv, dim=1) for t in (k, v))
            p = torch.softmax(torch.einsum("hd,nhd->hn", q[r, 0].float(), kr) / d ** 0.5, dim=-1)
            want[r] = torch.einsum("hn,nhd->hd", p, vr)
        assert rel_row_err(out.cpu().numpy(), want.numpy()) <= 2e-3
        assert torch.equal(ln.cpu(), (lens + step + 1).to(torch.int32))
    assert torch.equal(kc.cpu().view(torch.int16), k.view(torch.int16))
    assert torch.equal(vc.cpu().view(torch.int16), v.view(torch.int16))

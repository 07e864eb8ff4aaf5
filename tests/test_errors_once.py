"""A CUDA error is reported by the call that met it and by no later one."""
import pytest
import torch

import paper_2503_23956_b200 as ac

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_an_error_is_not_reported_again():
    """aircache_check_status synchronises, which a stream that is being captured does not allow: an error of the host side.
    The append behind it has nothing to do with it."""
    layers, hkv, d, slack = 2, 2, 64, 2
    sh = ac.shape(layers, 1, 4, hkv, d, 8, 4, 2, slack)
    ws = torch.zeros(ac.aircache_workspace_bytes(sh), dtype=torch.uint8, device=DEV)
    lens = torch.tensor([3, 1], dtype=torch.int32, device=DEV)
    offsets = torch.tensor([0, 3 + slack, 4 + 2 * slack], dtype=torch.int64, device=DEV)
    rows = 4 + 2 * slack
    k, v = (torch.zeros((rows, hkv, d), dtype=torch.bfloat16, device=DEV) for _ in range(2))
    new = torch.ones((layers, 1, hkv, d), dtype=torch.bfloat16, device=DEV)
    cache = ac.ragged_view(k, v, offsets, lens, rows)
    torch.cuda.synchronize()
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(stream):
        graph.capture_begin()
        met = ac.aircache_check_status(ws, stream, check=False)
        try:
            graph.capture_end()
        except RuntimeError:
            pass   # the capture was spoilt
    assert met == ac.ERR_CUDA
    assert ac.aircache_append(sh, cache, new, new, 0, check=False) == ac.OK
    torch.cuda.synchronize()
    assert lens.tolist() == [4, 2] and bool((k[3] == 1).all()) and bool((v[6] == 1).all())

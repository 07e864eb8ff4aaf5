"""A program that ends its context (cudaDeviceReset) and goes on with a new one: what the library keeps of a context - limits
of its kernels, the address of its built-in array - must not outlive it.  In a process of its own, with the runtime's
allocator and no torch tensors, since torch's would be lost with the context."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
import ctypes as C, glob, os, sys
import torch
import paper_2503_23956_b200 as ac

found = glob.glob(os.path.join(os.path.dirname(torch.__file__), "..", "nvidia", "cuda_runtime", "lib", "libcudart.so*"))
rt = C.CDLL(sorted(found)[-1] if found else "/usr/local/cuda/lib64/libcudart.so")


class Buffer:
    def __init__(self, n):
        p = C.c_void_p()
        assert rt.cudaMalloc(C.byref(p), C.c_size_t(n)) == 0 and rt.cudaMemset(p, 0, C.c_size_t(n)) == 0
        self.p, self.n = p.value, n

    def data_ptr(self):
        return self.p

    def numel(self):
        return self.n

    def element_size(self):
        return 1


def chain(L, hkv, alpha):
    hq, d, nv, nt, w, slack = 4 * hkv, 128, 300, 20, 16, 2
    sh = ac.shape(L, 1, hq, hkv, d, nv, nt, w, slack)
    ws, k = Buffer(ac.aircache_workspace_bytes(sh)), Buffer(L * hkv * (nv + nt) * d * 2)
    full = ac.Full(k.p, k.p, hkv * (nv + nt) * d, hkv * (nv + nt) * d, (nv + nt) * d, d)
    rows = ac.aircache_total_rows(sh, 0.2)
    kc, vc, off, lens, bud = (Buffer(n) for n in (rows * hkv * d * 2, rows * hkv * d * 2, (L + 1) * 8, L * 4, L * 4))
    cache = ac.Ragged(kc.p, vc.p, off.p, lens.p, rows, 0)
    q, new, out, scores = Buffer(L * hq * d * 2), Buffer(L * hkv * d * 2), Buffer(L * hq * d * 4), Buffer(L * nv * 4)
    qw = Buffer(L * w * hq * d * 2)
    ac.aircache_reset_status(ws, 0)
    ac.aircache_score(sh, full, qw, alpha, scores, None, ws, 0)
    ac.aircache_budget(sh, scores, 0.2, 0, bud, None, None, cache, ws, 0)
    ac.aircache_compact(sh, full, scores, bud, 0.2, cache, None, ws, 0)
    ac.aircache_decode_attn(sh, cache, q, out, ws, 0)
    ac.aircache_decode_step(sh, cache, q, new, new, 0, out, ws, 0)
    ac.aircache_decode_attn_static(sh, cache, q, out, 0)
    ac.aircache_check_status(ws, 0)


for turn in range(3):
    for L, hkv, alpha in ((3, 2, 0.9), (80, 4, 0.0), (12, 1, 0.9)):
        chain(L, hkv, alpha)
    assert rt.cudaDeviceSynchronize() == 0 and rt.cudaDeviceReset() == 0
print("three contexts")
"""


def test_calls_in_a_new_context():
    res = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert res.returncode == 0 and "three contexts" in res.stdout, res.stderr[-2000:]

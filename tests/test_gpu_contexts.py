"""Calls in several CUDA contexts of one process: what the library remembers between calls belongs to a context (shared-memory limits
of kernels, the address of the built-in scratch) and must not be taken from one that is gone.  Runs in a child process that makes
its contexts with the driver API."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes, sys
import numpy as np
import torch
import paper_2602_11562_b200 as P
from workloads import make_custom

cu, lib, mode = ctypes.CDLL("libcuda.so.1"), P.load_library(), sys.argv[1]
def ok(rc):
    assert rc == 0, rc
ok(cu.cuInit(0))
dev = ctypes.c_int()
ok(cu.cuDeviceGet(ctypes.byref(dev), 0))
bf16 = mode == "bf16"
# both need kernels with more than 48 KB of dynamic shared memory
w = make_custom(U=2, C=40, L=640, d=128, H=4, S=5 if not bf16 else 64, M=1, dtype="bf16" if bf16 else "f32", seed=91)
if mode == "static":
    w = make_custom(U=2, C=7, L=96, d=64, H=4, S=16, M=1, dtype="f32", seed=92)
s, dt = w.spec, torch.bfloat16 if bf16 else torch.float32
cfg = P.make_config(num_users=s.U, max_len=s.L, d_model=s.d, d_qk=w.Wq.shape[1], num_heads=s.H, seg_size=s.S, num_gsta_layers=s.M,
                    dtype=s.dtype, total_cands=w.N, max_cands_per_user=s.C)
host = [torch.from_numpy(np.ascontiguousarray(a)) for a in (w.items, w.lengths, w.cands, w.cand_offsets, w.Wq, w.Wk, w.Wv, w.Wg)]
host = [a.to(dt) if a.is_floating_point() else a.to(torch.int32) for a in host]

def one_call():
    ptrs = []
    def alloc(n):
        p = ctypes.c_void_p()
        ok(cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(n)))
        ptrs.append(p)
        return p
    args = []
    for a in host:
        p = alloc(a.numel() * a.element_size())
        ok(cu.cuMemcpyHtoD_v2(p, ctypes.c_void_p(a.data_ptr()), ctypes.c_size_t(a.numel() * a.element_size())))
        args.append(p.value)
    out = torch.zeros((w.N, s.n_seg, s.d) if mode == "static" else (w.N, s.d), dtype=dt)
    size = out.numel() * out.element_size()
    o = alloc(size)
    if mode == "static":
        ok(lib.laser_sta_forward_static(ctypes.byref(cfg), *args[:7], o, None, None))
    else:
        need = P.laser_workspace_bytes(cfg)
        ok(lib.laser_forward(ctypes.byref(cfg), *args, None, o, alloc(need), ctypes.c_size_t(need), None))
    ok(cu.cuCtxSynchronize())
    ok(cu.cuMemcpyDtoH_v2(ctypes.c_void_p(out.data_ptr()), o, ctypes.c_size_t(size)))
    for p in ptrs:
        ok(cu.cuMemFree_v2(p))
    return out

def context():
    c = ctypes.c_void_p()
    ok(cu.cuCtxCreate_v2(ctypes.byref(c), 0, dev))
    return c

first = context()
a = one_call()
second = context()                       # beside the first, on the same device
b = one_call()
ok(cu.cuCtxDestroy_v2(second))
ok(cu.cuCtxDestroy_v2(first))
third = context()                        # both gone
c = one_call()
ok(cu.cuCtxDestroy_v2(third))
assert torch.isfinite(a.float()).all() and a.float().abs().max() > 0
assert torch.equal(a, b) and torch.equal(a, c)
print("contexts ok")
"""


@pytest.mark.parametrize("mode", ["f32", "bf16", "static"])
def test_calls_in_several_contexts_agree(mode, repo_root):
    env = dict(os.environ, PYTHONPATH=repo_root)
    r = subprocess.run([sys.executable, "-c", CHILD, mode], cwd=repo_root, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "contexts ok" in r.stdout, (r.stdout[-2000:], r.stderr[-2000:])

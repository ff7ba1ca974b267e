"""Solves in a context that may use part of the GPU only (a green context of 32 SMs): grids whose on-chip
launch needs more CTAs than fit at once are streamed instead, alone and in batches, with the same results
to the solves' accuracy.  In a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

SCRIPT = r"""
import ctypes, sys
import torch
from paper_2603_23343_gb300 import binding as B, inputs

shapes = [(32, 32, 32), (64, 64, 64), (64, 60, 62)]
bs = [torch.from_numpy(inputs.uniform_rhs(s, 500 + i)).double().cuda() for i, s in enumerate(shapes)]
batch = [bs[1], bs[1], bs[0], bs[0]]
ws = [B.alloc_workspace(s, io_dtype=B.F64) for s in shapes]


def solves():
    out = []
    for b, w in zip(bs, ws):
        for mode in ("graph", "host_loop"):
            out.append(B.pcg_solve(b, tol=1e-6, workspace=w, mode=mode))
    for graph in (False, True):
        xs, rs = B.pcg_solve_batched(batch, tol=1e-6, graph=graph)
        out += list(zip(xs, rs))
    torch.cuda.synchronize()
    return out


whole = solves()
cu = ctypes.CDLL("libcuda.so.1")


def call(name, *args):
    rc = getattr(cu, name)(*args)
    if rc:
        print("unavailable:", name, rc)
        sys.exit(7)


dev, n = ctypes.c_int(0), ctypes.c_uint(1)
sms, part = (ctypes.c_uint64 * 256)(), (ctypes.c_uint64 * 256)()  # CUdevResource, with room to spare
desc, green, ctx = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
call("cuDeviceGet", ctypes.byref(dev), 0)
call("cuDeviceGetDevResource", dev, sms, 1)
call("cuDevSmResourceSplitByCount", part, ctypes.byref(n), sms, None, 0, 32)
call("cuDevResourceGenerateDesc", ctypes.byref(desc), part, 1)
call("cuGreenCtxCreate", ctypes.byref(green), desc, dev, 1)
call("cuCtxFromGreenCtx", ctypes.byref(ctx), green)
call("cuCtxPushCurrent_v2", ctx)
partial = solves()
call("cuCtxPopCurrent_v2", ctypes.byref(ctypes.c_void_p()))
for (x, r), (y, q) in zip(whole, partial):
    assert r["status"] == q["status"] == B.OK and abs(r["iters"] - q["iters"]) <= 2, (r, q)
    assert float((x - y).norm()) <= 5e-5 * float(x.norm())
print("done")
"""


def test_a_context_of_part_of_the_gpu(gpu_lib):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    p = subprocess.run([sys.executable, "-c", SCRIPT], capture_output=True, text=True, timeout=120, cwd=root,
                       env={**os.environ, "PYTHONPATH": root})
    if p.returncode == 7:
        pytest.skip(p.stdout.strip())
    assert p.returncode == 0 and p.stdout.strip() == "done", (p.stdout[-500:], p.stderr[-1500:])

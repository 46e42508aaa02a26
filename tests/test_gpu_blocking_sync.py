"""A process that asks CUDA for blocking synchronisation gets it in the solve: its thread
sleeps while the iterations run, and x is the same bit for bit as with the busy poll."""

import json
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import ctypes, hashlib, json, sys, time
if int(sys.argv[1]):
    cu = ctypes.CDLL("libcuda.so.1")
    assert cu.cuInit(0) == 0
    assert cu.cuDevicePrimaryCtxSetFlags_v2(0, 4) == 0          # CU_CTX_SCHED_BLOCKING_SYNC
import torch
from paper_2405_05865_gb300 import Context
ctx = Context(0)
g = torch.Generator(device="cuda").manual_seed(3)
A = ctx.rbf_kernel(torch.rand((8192, 3), generator=g, device="cuda", dtype=torch.float64), 0.1)
b = torch.randn(8192, generator=g, device="cuda", dtype=torch.float64)
f = ctx.nystrom(ctx.sketch(A, 256, 8), 1e-2, phi=0)
for _ in range(2):
    torch.cuda.synchronize()
    w, c = time.monotonic(), time.thread_time()
    x, info = ctx.solve(f, A, b, 1e-2, tol=1e-10, max_inner=0, check_every=32)
    w, c = time.monotonic() - w, time.thread_time() - c
print(json.dumps(dict(wall=w, cpu=c, status=info["status"], iters=info["outer_iters"],
                      x=hashlib.sha256(x.cpu().numpy().tobytes()).hexdigest())))
"""


def _run(blocking):
    p = subprocess.run([sys.executable, "-c", CHILD, str(int(blocking))], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    return json.loads(p.stdout.strip().splitlines()[-1])


def test_blocking_sync_sleeps():
    poll, block = _run(False), _run(True)
    assert poll["status"] == block["status"] == 0
    assert poll["x"] == block["x"] and poll["iters"] == block["iters"] > 100
    # issuing the launches is left to the thread; a busy poll takes all of the time
    assert block["cpu"] < 0.7 * block["wall"], block

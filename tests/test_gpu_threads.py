"""First calls from several threads at once: kernel attributes are set per process, and no thread may launch before they are; a thread
that has called nothing of CUDA yet has no context, which the driver's tensor-map call wants."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import threading
import torch
from paper_2512_24545_b200 import inputs, mdbf as M
from helpers import GpuLayer

spec = inputs.scaled(inputs.qproj(1664), name="threads", d_out=640, d_in=1024, k=512, l=16)
kinds = [(1, M.KERNEL_AUTO), (1, M.KERNEL_I8), (8, M.KERNEL_AUTO), (200, M.KERNEL_AUTO), (8, M.KERNEL_ALU), (200, M.KERNEL_PREFILL)]
jobs = []
for T, kernel in kinds:
    for copy in range(3):
        g = GpuLayer(spec, 200)
        M.mdbf_set_kernel(g.h, kernel)
        x = torch.randn(T, 1024, generator=torch.Generator(device="cuda").manual_seed(T), device="cuda").to(torch.bfloat16)
        jobs.append((g, x, torch.zeros(T, 640, dtype=torch.bfloat16, device="cuda"), torch.cuda.Stream()))
torch.cuda.synchronize()
start, errors = threading.Barrier(len(jobs)), []

def work(g, x, y, stream):
    try:
        start.wait()
        M.mdbf_linear_forward(g.h, x.data_ptr(), y.data_ptr(), x.shape[0], M.BF16, stream.cuda_stream)
    except Exception as e:
        errors.append(repr(e))

threads = [threading.Thread(target=work, args=j) for j in jobs]
for t in threads: t.start()
for t in threads: t.join()
torch.cuda.synchronize()
assert not errors, errors
for i, (g, x, y, _) in enumerate(jobs):
    again = torch.zeros_like(y)
    M.mdbf_linear_forward(g.h, x.data_ptr(), again.data_ptr(), x.shape[0], M.BF16, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert M.mdbf_poll_status(g.h) == 0
    assert torch.equal(y, again) and float(y.float().abs().max()) > 0, kinds[i // 3]
print("threads ok")
"""

QUANTIZER = r"""
import threading
import numpy as np
import torch
from paper_2512_24545_b200 import inputs, mdbf as M
torch.zeros(1, device="cuda")
Z = torch.from_numpy(inputs.make_factor_matrix(300, 256, seed=3)).cuda()
Q0 = torch.from_numpy(inputs.make_start_block(256, 8, seed=3)).cuda()
n = M.mdbf_msvid_workspace_bytes(300, 256, 8)
jobs = [[torch.zeros(300, 8, dtype=torch.int32, device="cuda"), torch.zeros(300, 8, device="cuda"), torch.zeros(256, 8, device="cuda"), torch.zeros(8, device="cuda"),
         torch.empty(n, dtype=torch.uint8, device="cuda"), torch.cuda.Stream()] for _ in range(6)]
torch.cuda.synchronize()
start, errors = threading.Barrier(len(jobs)), []

def work(S, U, V, s, ws, stream):
    try:
        start.wait()
        M.mdbf_msvid(Z.data_ptr(), 300, 256, 8, 4, Q0.data_ptr(), S.data_ptr(), U.data_ptr(), V.data_ptr(), s.data_ptr(), ws.data_ptr(), n, stream.cuda_stream)
    except Exception as e:
        errors.append(repr(e))

threads = [threading.Thread(target=work, args=j) for j in jobs]
for t in threads: t.start()
for t in threads: t.join()
torch.cuda.synchronize()
assert not errors, errors
for j in jobs[1:]:
    assert all(torch.equal(a, b) for a, b in zip(j[:4], jobs[0][:4]))
assert bool(torch.isfinite(jobs[0][3]).all()) and float(jobs[0][3][0]) > 0
print("threads ok")
"""


@pytest.mark.parametrize("child", [CHILD, QUANTIZER], ids=["forward", "quantizer"])
def test_first_calls_of_several_threads(child):
    from paper_2512_24545_b200 import build
    build.build()
    here = os.path.dirname(os.path.abspath(__file__))
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([here, os.path.dirname(here)]))
    p = subprocess.run([sys.executable, "-c", child], env=env, cwd=os.path.dirname(here), capture_output=True, text=True, timeout=300)
    assert p.returncode == 0 and "threads ok" in p.stdout, p.stdout + p.stderr

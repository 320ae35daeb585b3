"""The library's first calls in a process come from several threads at once: what it looks up once (the tensor-map encoder, the number of
SMs, the kernels' shared-memory limits) is there for each of them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import threading, torch
from paper_2605_16732_b200 import binding as dq
K, N, M, n = 128, 64, 32, 16
torch.manual_seed(0)
Q = torch.linalg.qr(torch.randn(K, K, device="cuda", dtype=torch.float64))[0].contiguous()
W, x = torch.randn(K, N, device="cuda"), torch.randn(M, K, device="cuda").to(torch.bfloat16)
ys, errors, gate = [torch.empty(M, N, dtype=torch.bfloat16, device="cuda") for _ in range(n)], [], threading.Barrier(n)
dq.lib()
torch.cuda.synchronize()
def work(i):
    try:
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            gate.wait()
            layer = dq.dirotq_prepare_layer(W, Q, 16, 64)
            ws = dq.alloc_workspace(layer, M)
            dq.dirotq_linear(x, layer, ys[i], ws)
            assert dq.dirotq_workspace_status(ws) == 0
    except Exception as e:
        errors.append(e)
threads = [threading.Thread(target=work, args=(i,)) for i in range(n)]
[t.start() for t in threads]
[t.join() for t in threads]
torch.cuda.synchronize()
assert not errors, errors
assert all(torch.equal(y, ys[0]) for y in ys)
"""


def test_first_calls_from_many_threads():
    for _ in range(3):
        r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]

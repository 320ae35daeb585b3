"""What the wait counters of the INT4 second kernels contain: a role's waits in its own kernel, not what was left of the kernel before it."""
import json
import os
import subprocess
import sys

import pytest
import torch

from paper_2605_16732_b200 import binding as dq

pytestmark = pytest.mark.gpu


def _counters(plan, parts):
    # a rotation of few, long tiles (twice the second kernel's time): that kernel's blocks are there for most of it, on other SMs
    M, K, N, r = 256, 6144, 256, 4096
    g = torch.Generator(device="cuda").manual_seed(plan)
    layer = dq.dirotq_prepare_layer(torch.randn(K, N, generator=g, device="cuda") * 0.02, torch.eye(K, device="cuda"), r, 64)
    x = torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16)
    y = torch.empty(M, N, dtype=torch.bfloat16, device="cuda")
    ws = dq.alloc_workspace(layer, M)
    dq.dirotq_set_rotation_tile(3)
    dq.dirotq_set_gemm_tile(plan)
    try:
        for i in range(3):
            if i == 1:  # (the first call of a kernel loads it)
                torch.cuda.synchronize()
                ws[:256].zero_()
                torch.cuda.synchronize()
            if parts:
                dq.dirotq_rotate_quantize(x, layer, ws)
                dq.dirotq_w4a4_gemm(M, layer, ws, y)
            else:
                dq.dirotq_linear(x, layer, y, ws)
        c = dq.dirotq_workspace_wait_counters(ws)
    finally:
        dq.dirotq_set_rotation_tile(0)
        dq.dirotq_set_gemm_tile(0)
    assert dq.dirotq_workspace_status(ws) == 0
    layer.close()
    return c


@pytest.mark.parametrize("parts", [False, True])  # dirotq_linear; its two parts, whose second one may not load weights early
@pytest.mark.parametrize("plan", [32, 64, 128, 130, 192, 256])
def test_waits_leave_the_previous_kernel_out(plan, parts):
    c = _counters(plan, parts)
    # Every role waits between the end of the previous kernel and its own end; the MMA role's total is that span.  A quarter more for the early
    # weights' first loads (some 3000 cycles of 25000 or more).
    assert c["unpack_wait_tma"] <= 1.25 * c["mma_role_total"], c
    assert c["epilogue_wait_accumulator"] <= c["epilogue_total"] <= 1.25 * c["mma_role_total"], c
    assert c["mma_wait_operands"] + c["mma_wait_accumulator"] <= c["mma_role_total"], c


PROGRAM = """
import json
from paper_2605_16732_b200 import binding as dq, build
dq.use_library(build.build_trace())
from test_gpu_wait_counters import _counters
print(json.dumps([_counters(plan, False) for plan in (32, 64, 128, 130, 192, 256)]))
"""


def test_the_diagnostic_build_counts_every_wait():
    here = os.path.dirname(os.path.abspath(__file__))
    r = subprocess.run([sys.executable, "-c", PROGRAM], capture_output=True, text=True, timeout=300, cwd=os.path.dirname(here),
                       env=dict(os.environ, PYTHONPATH=os.pathsep.join([os.path.dirname(here), here])))
    assert r.returncode == 0, r.stderr[-2000:]
    for c in json.loads(r.stdout):
        # a kernel's first activations are waited for by everyone; nothing waits for scales by themselves
        assert min(c["mma_wait_operands"], c["unpack_wait_tma"], c["epilogue_wait_accumulator"]) > 0 and c["epilogue_wait_scales"] == 0, c
        assert c["unpack_wait_tma"] <= 1.25 * c["mma_role_total"] and c["epilogue_wait_accumulator"] <= c["epilogue_total"], c
        assert c["mma_wait_operands"] + c["mma_wait_accumulator"] <= c["mma_role_total"], c

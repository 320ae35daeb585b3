"""The W4A8 second kernel in CTA pairs (256 token rows, 128 or 256 columns): the edges of its tiles against the oracle, and the same bits
as single CTAs where a pair takes several tiles (the integer sums are exact, so the plan must not show)."""
import pytest
import torch

import test_gpu_w4a8
from paper_2605_16732_b200 import binding as dq
from paper_2605_16732_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture
def plan(request):
    dq.dirotq_set_gemm_tile(request.param)
    yield request.param
    dq.dirotq_set_gemm_tile(0)


@pytest.mark.parametrize("plan", [256, 512], indirect=True)
@pytest.mark.parametrize("M, N", [(1, 96), (129, 160), (257, 400)])  # second CTA without rows; ragged columns; second half without columns
def test_parity_at_tile_edges(plan, M, N):
    spec = synth.LayerSpec(K=256, N=N, r=32, G=64, model=synth.PIXART, seed=11, calib_tokens=512)
    test_gpu_w4a8._run_case(spec, M=M)


def test_same_bits_as_single_ctas():
    M, K, N, r = 4173, 1152, 1408, 128  # several tiles per pair, ragged rows, two rank-r chunks
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16)
    Q = torch.linalg.qr(torch.randn(K, K, generator=g, device="cuda", dtype=torch.float64))[0].float().contiguous()
    W = torch.randn(K, N, generator=g, device="cuda") * 0.02
    layer = dq.dirotq_prepare_layer_w4a8(W, Q, r)
    ws = dq.alloc_workspace(layer, M)
    outs = []
    try:
        for columns in (128, 256, 512, 0):
            dq.dirotq_set_gemm_tile(columns)
            outs.append(torch.empty(M, N, dtype=torch.bfloat16, device="cuda"))
            dq.dirotq_linear(x, layer, outs[-1], ws)
    finally:
        dq.dirotq_set_gemm_tile(0)
    assert dq.dirotq_workspace_status(ws) == 0
    assert all(torch.equal(o.view(torch.int16), outs[0].view(torch.int16)) for o in outs[1:])
    layer.close()

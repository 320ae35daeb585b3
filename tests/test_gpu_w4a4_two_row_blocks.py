"""The grouped INT4 second kernel with tiles of 256 token rows, in CTA pairs (258: x 256 columns) and in one CTA (130: x 128 columns): the edges
of the tiles against the oracle, and the same bits as the other plans where a CTA takes several tiles (each output element is
accumulated in the same order)."""
import pytest
import torch

import test_gpu_asym
import test_gpu_parity
from paper_2605_16732_b200 import binding as dq
from paper_2605_16732_b200 import synth

pytestmark = pytest.mark.gpu
PLANS = [258, 130, 512]  # (512 names no plan of this kernel: it chooses for itself)


@pytest.fixture
def plan(request):
    dq.dirotq_set_gemm_tile(request.param)
    yield request.param
    dq.dirotq_set_gemm_tile(0)


# second row block without rows; ragged columns; second half of the columns without any; an odd number of groups (K - r = 560 and 480)
@pytest.mark.parametrize("plan", [*PLANS, 32], indirect=True)  # (32: 32-column tiles, ragged here too)
@pytest.mark.parametrize("M, K, N, r, G", [(1, 512, 96, 16, 64), (129, 576, 160, 16, 64), (257, 512, 400, 32, 128), (300, 640, 272, 128, 64)])
def test_parity_at_tile_edges(plan, M, K, N, r, G):
    spec = synth.LayerSpec(K=K, N=N, r=r, G=G, model=synth.PIXART, seed=71, calib_tokens=512)
    test_gpu_parity._run_case(spec, M=M, check_rot=False)


@pytest.mark.parametrize("plan", PLANS, indirect=True)
def test_parity_asymmetric_codes(plan):
    spec = synth.LayerSpec(K=640, N=400, r=32, G=64, model=synth.PIXART, seed=72, calib_tokens=512)
    test_gpu_asym._run_case(spec, M=200, shift=1.5)


@pytest.mark.parametrize("G, r", [(64, 32), (128, 128), (64, 464)])  # one, two and eight rank-r chunks; odd and even numbers of groups
def test_same_bits_as_other_tiles(G, r):
    M, K, N = 4173, 1152, 4736  # several tiles per CTA under every plan, ragged rows and columns
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16)
    Q = torch.linalg.qr(torch.randn(K, K, generator=g, device="cuda", dtype=torch.float64))[0].float().contiguous()
    W = torch.randn(K, N, generator=g, device="cuda") * 0.02
    layer = dq.dirotq_prepare_layer(W, Q, r, G)
    ws = dq.alloc_workspace(layer, M)
    outs = []
    try:
        for columns in (256, 0, 32, 64, 128, 192, *PLANS):
            dq.dirotq_set_gemm_tile(columns)
            outs.append(torch.empty(M, N, dtype=torch.bfloat16, device="cuda"))
            dq.dirotq_linear(x, layer, outs[-1], ws)
    finally:
        dq.dirotq_set_gemm_tile(0)
    assert dq.dirotq_workspace_status(ws) == 0
    assert all(torch.equal(o.view(torch.int16), outs[0].view(torch.int16)) for o in outs[1:])
    layer.close()

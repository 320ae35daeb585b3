"""The INT4 second kernels load and expand the first stages' weights while the call's first stage is still running: calls of fewer, as many and more
k-blocks than a ring has stages, one and several tiles per CTA, against the same call in two parts (whose second part does not); bit for bit."""
import pytest
import torch

from paper_2605_16732_b200 import binding as dq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("plan", [32, 64, 66, 128, 130, 192, 256, 258, 512])
@pytest.mark.parametrize("M, K, N, r, G", [(5, 256, 48, 16, 64), (130, 512, 400, 32, 64), (300, 768, 272, 64, 64), (257, 1024, 320, 128, 128), (1500, 1664, 2832, 32, 64)])
def test_linear_equals_its_two_parts(plan, M, K, N, r, G):
    g = torch.Generator(device="cuda").manual_seed(K + plan)
    Q = torch.linalg.qr(torch.randn(K, K, generator=g, device="cuda", dtype=torch.float64))[0].float().contiguous()
    layers = [dq.dirotq_prepare_layer(torch.randn(K, N, generator=g, device="cuda") * 0.02, Q, r, G) for _ in range(2)]
    x = [torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2)]
    ws = dq.alloc_workspace(layers[0], M)
    ys = torch.empty(2, 2, M, N, dtype=torch.bfloat16, device="cuda")
    dq.dirotq_set_gemm_tile(plan)
    try:
        for i in (0, 1):
            dq.dirotq_rotate_quantize(x[i], layers[i], ws)
            dq.dirotq_w4a4_gemm(M, layers[i], ws, ys[0, i])
        torch.cuda.synchronize()
        for _ in range(3):  # back to back, so that every kernel starts under the previous one
            for i in (0, 1):
                dq.dirotq_linear(x[i], layers[i], ys[1, i], ws)
    finally:
        dq.dirotq_set_gemm_tile(0)
    assert dq.dirotq_workspace_status(ws) == 0
    assert torch.equal(ys[0].view(torch.int16), ys[1].view(torch.int16))
    for layer in layers:
        layer.close()

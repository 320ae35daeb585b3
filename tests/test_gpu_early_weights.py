"""The INT4 second kernels load and expand the first stages' weights while the call's first stage is still running: calls of fewer, as many and more
k-blocks than a ring has stages, one and several tiles per CTA, all three formats, chosen plans and captured graphs, against the same call in two
parts (whose second part does not); bit for bit."""
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


def _pair(fmt, K, N, r, g):
    """Two layers of one shape."""
    Q = torch.linalg.qr(torch.randn(K, K, generator=g, device="cuda", dtype=torch.float64))[0].contiguous()
    W = [torch.randn(K, N, generator=g, device="cuda") * 0.02 for _ in range(2)]
    if fmt == "int4_ph":
        return [dq.dirotq_prepare_layer_ph(w, Q[:, :r].contiguous(), 64) for w in W]
    return [(dq.dirotq_prepare_layer_asym if fmt == "int4_asym" else dq.dirotq_prepare_layer)(w, Q, r, 64) for w in W]


# projection form: two kernels before the second one, and three (K = 2048: the first step's reduction is split); the plan that the call chooses;
# the rotation in 64- and 128-column tiles and CTA pairs
@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("fmt, rotation, plans", [("int4", 0, (0,)), ("int4", 5, (0, 32)), ("int4", 1, (64, 258)), ("int4_asym", 0, (0, 64, 130, 192)),
                                                  ("int4_ph", 0, (0, 32, 64, 128, 130, 192, 256, 258))])
@pytest.mark.parametrize("M, K, N, r", [(5, 512, 48, 16), (130, 2048, 400, 32), (1500, 1664, 2832, 32)])
def test_formats_chosen_plans_and_graphs(M, K, N, r, fmt, rotation, plans, captured):
    g = torch.Generator(device="cuda").manual_seed(K + rotation)
    layers = _pair(fmt, K, N, r, g)
    x = [torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2)]
    ws = dq.alloc_workspace(layers[0], M)
    ys = torch.zeros(2, 2, M, N, dtype=torch.bfloat16, device="cuda")
    dq.dirotq_set_rotation_tile(rotation)
    try:
        for plan in plans:
            dq.dirotq_set_gemm_tile(plan)
            for i in (0, 1):
                dq.dirotq_rotate_quantize(x[i], layers[i], ws)
                torch.cuda.synchronize()
                dq.dirotq_w4a4_gemm(M, layers[i], ws, ys[0, i])
                torch.cuda.synchronize()

            def calls():
                for _ in range(3):
                    for i in (0, 1):
                        dq.dirotq_linear(x[i], layers[i], ys[1, i], ws)
            ys[1].zero_()
            if captured:
                calls()  # (a kernel's first call loads it)
                torch.cuda.synchronize()
                ys[1].zero_()
                graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
                with torch.cuda.graph(graph, stream=side):
                    calls()
                graph.replay()
                graph.replay()
            else:
                calls()
            assert dq.dirotq_workspace_status(ws) == 0
            assert torch.equal(ys[0].view(torch.int16), ys[1].view(torch.int16)), plan
    finally:
        dq.dirotq_set_rotation_tile(0)
        dq.dirotq_set_gemm_tile(0)
    for layer in layers:
        layer.close()


@pytest.mark.parametrize("fmt", ["int4", "int4_asym", "int4_ph"])
def test_call_right_behind_its_preparation(fmt):
    """The weights that are loaded early were written by the kernel before the call's first one; nothing waits between the two."""
    M, K, N, r = 64, 768, 1024, 32
    g = torch.Generator(device="cuda").manual_seed(8)
    x = torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16)
    for layer in _pair(fmt, K, N, r, g):  # (loads every kernel)
        ws = dq.alloc_workspace(layer, M)
        dq.dirotq_linear(x, layer, torch.empty(M, N, dtype=torch.bfloat16, device="cuda"), ws)
        layer.close()
    W, Q = torch.randn(K, N, generator=g, device="cuda") * 0.02, torch.eye(K, device="cuda", dtype=torch.float64)
    y = torch.empty(2, M, N, dtype=torch.bfloat16, device="cuda")
    torch.cuda.synchronize()
    layer = dq.dirotq_prepare_layer_ph(W, Q[:, :r].contiguous(), 64) if fmt == "int4_ph" else \
        (dq.dirotq_prepare_layer_asym if fmt == "int4_asym" else dq.dirotq_prepare_layer)(W, Q, r, 64)
    dq.dirotq_linear(x, layer, y[0], ws)
    torch.cuda.synchronize()
    dq.dirotq_linear(x, layer, y[1], ws)
    assert dq.dirotq_workspace_status(ws) == 0
    assert torch.equal(y[0].view(torch.int16), y[1].view(torch.int16))
    layer.close()

"""Calls of fewer than 128 token rows load only the rows that exist (in eights): every format gives the bits that the same tokens get in a call of 128
rows, whatever the workspace and the SMs' shared memory held before (here: NaN activations of another call)."""
import pytest
import torch

from paper_2605_16732_b200 import binding as dq

pytestmark = pytest.mark.gpu


def _layer(fmt, W, Q, r):
    if fmt == "int4":
        return dq.dirotq_prepare_layer(W, Q, r, 64)
    if fmt == "int4_g128":
        return dq.dirotq_prepare_layer(W, Q, r, 128)
    if fmt == "int4_asym":
        return dq.dirotq_prepare_layer_asym(W, Q, r, 64)
    if fmt == "w4a8":
        return dq.dirotq_prepare_layer_w4a8(W, Q, r)
    if fmt == "nvfp4":
        return dq.dirotq_prepare_layer_nvfp4(W, Q, r, -6)
    Uh = Q[:, :r].contiguous()
    return dq.dirotq_prepare_layer_ph(W, Uh, 64) if fmt == "int4_ph" else dq.dirotq_prepare_layer_nvfp4_ph(W, Uh, -6)


@pytest.mark.parametrize("plan", [0, 64, 128, 192, 256])
@pytest.mark.parametrize("fmt", ["int4", "int4_g128", "int4_asym", "w4a8", "nvfp4", "int4_ph", "nvfp4_ph"])
def test_same_bits_as_in_a_full_row_block(fmt, plan):
    K, N, r = 768, 400, 32
    g = torch.Generator(device="cuda").manual_seed(5)
    Q = torch.linalg.qr(torch.randn(K, K, generator=g, device="cuda", dtype=torch.float64))[0].contiguous()
    layer = _layer(fmt, torch.randn(K, N, generator=g, device="cuda") * 0.02, Q, r)
    x = torch.randn(128, K, generator=g, device="cuda").to(torch.bfloat16)
    ws = dq.alloc_workspace(layer, 128)
    full, y, spoil = (torch.empty(128, N, dtype=torch.bfloat16, device="cuda") for _ in range(3))
    dq.dirotq_set_gemm_tile(plan)
    try:
        dq.dirotq_linear(x, layer, full, ws)
        for M in (1, 7, 8, 9, 31, 64, 121, 127):
            dq.dirotq_linear(torch.full_like(x, float("nan")), layer, spoil, ws)
            dq.dirotq_linear(x[:M].contiguous(), layer, y[:M], ws)
            assert torch.equal(y[:M].view(torch.int16), full[:M].view(torch.int16)), M
    finally:
        dq.dirotq_set_gemm_tile(0)
    assert dq.dirotq_workspace_status(ws) == 0
    layer.close()


@pytest.mark.parametrize("plan", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("fmt", ["int4", "int4_g128", "int4_asym", "w4a8", "nvfp4"])  # (the projection form's first stage has one plan)
def test_same_bits_under_every_rotation_plan(fmt, plan):
    dq.dirotq_set_rotation_tile(plan)
    try:
        test_same_bits_as_in_a_full_row_block(fmt, 0)
    finally:
        dq.dirotq_set_rotation_tile(0)

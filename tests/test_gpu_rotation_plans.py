"""The rotation plan chosen by default on long main loops (CTA pairs from 6144 columns on) gives the bits of the 128 x 256 plan, in every
format: one turn and several, an odd number of row blocks, ragged rows."""
import pytest
import torch

from paper_2605_16732_b200 import binding as dq

pytestmark = pytest.mark.gpu

K, N, R = 6144, 64, 32


@pytest.fixture(scope="module")
def rotation():
    g = torch.Generator(device="cuda").manual_seed(2)
    v = torch.randn(K, generator=g, device="cuda", dtype=torch.float64)
    v /= v.norm()
    return torch.eye(K, device="cuda", dtype=torch.float64) - 2.0 * torch.outer(v, v)


@pytest.mark.parametrize("fmt", ["int4", "int4_g128", "int4_asym", "w4a8", "nvfp4"])
@pytest.mark.parametrize("M", [512, 700, 1400])
def test_default_plan_against_single_ctas(rotation, fmt, M):
    g = torch.Generator(device="cuda").manual_seed(M)
    W = 0.02 * torch.randn(K, N, generator=g, device="cuda")
    x = torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16)
    layer = {"int4": lambda: dq.dirotq_prepare_layer(W, rotation, R, 64), "int4_g128": lambda: dq.dirotq_prepare_layer(W, rotation, R, 128),
             "int4_asym": lambda: dq.dirotq_prepare_layer_asym(W, rotation, R, 64), "w4a8": lambda: dq.dirotq_prepare_layer_w4a8(W, rotation, R),
             "nvfp4": lambda: dq.dirotq_prepare_layer_nvfp4(W, rotation, R, 0)}[fmt]()
    outs = []
    try:
        for plan in (2, 0):
            dq.dirotq_set_rotation_tile(plan)
            ws = dq.alloc_workspace(layer, M)
            dq.dirotq_rotate_quantize(x, layer, ws)
            assert dq.dirotq_workspace_status(ws) == 0
            outs.append(ws[256:].clone())  # behind the status block: codes, scales, 16-bit coefficients
    finally:
        dq.dirotq_set_rotation_tile(0)
    assert torch.equal(outs[0], outs[1])
    layer.close()

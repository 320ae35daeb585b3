"""Row counts that fill no tile: a call with padding rows does not take longer than the call with those rows filled (the padding's zeros
used to go through the quantizer's path for zero scales, which divides), and the rows that are there come out the same."""
import pytest
import torch

from paper_2605_16732_b200 import binding as dq

pytestmark = pytest.mark.gpu


def _time(fn, calls=50):
    fn()
    best = float("inf")
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda._sleep(4_000_000)  # the calls are queued while this runs: the device's time is measured, not the host's
        a.record()
        for _ in range(calls):
            fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("plan", [1, 2, 4, 5])
@pytest.mark.parametrize("asym", [False, True])
def test_padding_rows(asym, plan):
    K, N, R, rows, full = 512, 64, 32, 1825, 2048
    g = torch.Generator(device="cuda").manual_seed(4)
    Q = torch.linalg.qr(torch.randn(K, K, generator=g, device="cuda", dtype=torch.float64))[0].contiguous()
    prepare = dq.dirotq_prepare_layer_asym if asym else dq.dirotq_prepare_layer
    export = dq.dirotq_workspace_export_asym if asym else dq.dirotq_workspace_export
    layer = prepare(0.02 * torch.randn(K, N, generator=g, device="cuda"), Q, R, 64)
    x = torch.randn(full, K, generator=g, device="cuda").to(torch.bfloat16)
    ws, wsf = dq.alloc_workspace(layer, rows), dq.alloc_workspace(layer, full)
    try:
        dq.dirotq_set_rotation_tile(plan)
        t, tf = _time(lambda: dq.dirotq_rotate_quantize(x[:rows], layer, ws)), _time(lambda: dq.dirotq_rotate_quantize(x, layer, wsf))
        x[5] = 0  # a row that is there and is zero
        dq.dirotq_rotate_quantize(x[:rows], layer, ws)
        dq.dirotq_rotate_quantize(x, layer, wsf)
    finally:
        dq.dirotq_set_rotation_tile(0)
    for part, whole in zip(export(layer, rows, ws), export(layer, full, wsf)):
        assert torch.equal(part, whole[:rows])
    assert t < 1.4 * tf, (t, tf)
    layer.close()

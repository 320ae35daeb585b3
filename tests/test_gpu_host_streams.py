"""dirotq_linear_host on several streams and threads: calls of few rows do not make calls on other streams wait, more of them than the library
has copy streams for run too, and one that is being captured takes nothing from the others.  Bits as from dirotq_linear."""
import threading

import pytest
import torch

from paper_2605_16732_b200 import binding as dq

pytestmark = pytest.mark.gpu

K, N, R = 512, 384, 32


def _layer():
    g = torch.Generator(device="cuda").manual_seed(5)
    Q = torch.linalg.qr(torch.randn(K, K, generator=g, device="cuda", dtype=torch.float64))[0].contiguous()
    return dq.dirotq_prepare_layer(0.02 * torch.randn(K, N, generator=g, device="cuda"), Q, R, 64)


class Call:
    """One caller's buffers on a stream of its own; `y` is the device entry point's result."""

    def __init__(self, layer, M, seed=0):
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16)
        self.layer, self.ws, self.stream = layer, dq.alloc_workspace(layer, M), torch.cuda.Stream()
        self.x_dev, self.y_dev = torch.empty_like(x), torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
        self.x, self.out = x.cpu().pin_memory(), torch.zeros((M, N), dtype=torch.bfloat16).pin_memory()
        y = torch.empty_like(self.y_dev)
        dq.dirotq_linear(x, layer, y, self.ws)
        self.y = y.cpu()
        torch.cuda.synchronize()

    def run(self):
        dq.dirotq_linear_host(self.x, self.layer, self.out, self.x_dev, self.y_dev, self.ws, stream=self.stream)
        self.done = torch.cuda.Event()
        self.done.record(self.stream)

    def check(self):
        self.done.synchronize()
        assert torch.equal(self.out.view(torch.int16), self.y.view(torch.int16))
        assert dq.dirotq_workspace_status(self.ws, stream=self.stream) == 0
        self.out.zero_()


@pytest.mark.parametrize("M", [511, 512, 1000, 2047])
def test_row_chunks_of_short_calls(M):
    layer = _layer()
    c = Call(layer, M)
    for _ in range(2):
        c.run()
        c.check()
    layer.close()


@pytest.mark.parametrize("M", [1024, 2500])
def test_a_call_does_not_wait_for_a_short_one_on_another_stream(M):
    layer = _layer()
    for attempt in range(4):  # (two streams can share one of the device's queues by chance; then others are tried)
        waiting, free = Call(layer, 1024, 1), Call(layer, M, 2)
        for c in (waiting, free):  # first uses, so that nothing is loaded or created below
            c.run()
            c.check()
        with torch.cuda.stream(waiting.stream):
            torch.cuda._sleep(int(2e8))  # about 0.1 s
            gate = torch.cuda.Event()
            gate.record()
        waiting.run()
        free.run()
        free.check()
        independent = not gate.query()
        waiting.check()
        if independent:
            break
    assert independent, "the call waited for the other"
    layer.close()


def test_many_streams_at_once():
    layer = _layer()
    calls = [Call(layer, 600 + 150 * i, i) for i in range(12)]  # short and long ones
    for _ in range(3):
        for c in calls:
            c.run()
        for c in calls:
            c.check()
    layer.close()


def test_a_captured_call_and_others_meanwhile():
    layer = _layer()
    captured, other = Call(layer, 2500, 1), Call(layer, 2500, 2)
    for c in (captured, other):
        c.run()
        c.check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=captured.stream):
        dq.dirotq_linear_host(captured.x, layer, captured.out, captured.x_dev, captured.y_dev, captured.ws, stream=captured.stream)
        other.run()
    other.check()
    for _ in range(2):
        with torch.cuda.stream(captured.stream):
            graph.replay()
            captured.done.record()
        captured.check()
    layer.close()


def test_threads_on_their_own_streams_and_layers_that_come_and_go():
    def work(seed, errors):
        try:
            for round_ in range(3):
                layer = _layer()
                c = Call(layer, 512 + 300 * seed + round_, seed)
                for _ in range(5):
                    c.run()
                    c.check()
                layer.close()
        except Exception as e:  # noqa: BLE001 (reported by the main thread)
            errors.append(e)

    errors = []
    threads = [threading.Thread(target=work, args=(i, errors)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_prepare_on_another_stream():
    """The call's scratch, and a blob that starts cleared, come from the current stream: neither is touched from there while a busy stream
    still prepares the layer."""
    g = torch.Generator(device="cuda").manual_seed(8)
    Q = torch.linalg.qr(torch.randn(K, K, generator=g, device="cuda", dtype=torch.float64))[0].contiguous()
    W = 0.02 * torch.randn(K, N, generator=g, device="cuda")
    side = torch.cuda.Stream()

    def busy(s):
        with torch.cuda.stream(s):
            torch.cuda._sleep(int(4e7))  # about 20 ms

    for prepare, export in ((lambda **kw: dq.dirotq_prepare_layer(W, Q, R, 64, **kw), dq.dirotq_layer_export),
                            (lambda **kw: dq.dirotq_prepare_layer_nvfp4(W, Q, R, 0, **kw), dq.dirotq_layer_export_nvfp4)):
        plain = prepare()
        want = [t.clone() for t in export(plain) if isinstance(t, torch.Tensor)]
        torch.cuda.synchronize()
        for late in (side, torch.cuda.current_stream()):  # the preparing stream is behind, then the current one
            busy(late)
            layer = prepare(stream=side)
            junk = [torch.full((K * N,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(3)]  # where the scratch was
            torch.cuda.synchronize()
            got = [t for t in export(layer) if isinstance(t, torch.Tensor)]
            assert all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(got, want))
            layer.close()
            del junk
        plain.close()

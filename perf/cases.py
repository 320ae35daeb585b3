"""The work this library is timed on: calls of its public entry points as a program that serves a diffusion transformer makes
them, over the sizes, formats and options it is used with.

A case names the call ("call"), the layer's format ("fmt"), the number of token rows M, the layer K -> N, the rank r of its
16-bit part and the quantization group G (groups of the INT4 formats; the other formats have their own granularity and ignore it).

    linear   dirotq_linear: one quantized layer on activations that are on the GPU
    shared   dirotq_rotate_quantize once, then dirotq_w4a4_gemm for three layers that read the same activations (q, k, v)
    host     dirotq_linear_host: activations and result in pinned host memory
    prepare  dirotq_prepare_layer on fp32 weights (and dirotq_layer_export, which makes its result comparable): what loading a
             model pays per layer

Activations follow paper_2605_16732_b200/synth.py: unit-variance channels, a few outlier channels of 50 to 80 times their size, a
shared low-rank component.  The rotation's first r columns span the leading directions of such activations (outlier channels,
then the low-rank basis); the rest completes them to an orthogonal matrix.  That is what a calibrated rotation looks like,
without an eigendecomposition per call of prepare().
"""
import math

import torch

from paper_2605_16732_b200 import binding as dq
from paper_2605_16732_b200 import synth

FORMATS = ("int4", "int4_asym", "w4a8", "nvfp4", "int4_ph", "nvfp4_ph")


def _case(call, fmt, M, K, N, r, G=64, name=None):
    c = {"call": call, "fmt": fmt, "M": M, "K": K, "N": N, "r": r, "G": G}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the attention projection of a small model on one 16 x 16 latent: a few microseconds, launches count
        _case("linear", "int4", 256, 1152, 1152, 32, name="pixart_proj_m256_int4"),
        # the text tokens of a joint block through its fused q/k/v layer, asymmetric activation codes
        _case("linear", "int4_asym", 512, 3072, 9216, 32, name="flux_text_qkv_m512_asym"),
        # q, k and v of a block on one rotation, 4096 image tokens
        _case("shared", "int4", 4096, 1152, 1152, 32, name="pixart_qkv_shared_m4096_int4"),
        # 8-bit activations, a tenth of the coefficients in 16 bits, wide to narrow
        _case("linear", "w4a8", 4096, 4608, 1152, 464, name="pixart_mlp_down_m4096_w4a8"),
        # the benchmark's layers (4096 image + 512 text tokens)
        _case("linear", "int4", 4608, 3072, 9216, 32, name="flux_qkv_m4608_int4"),
        _case("linear", "int4", 4608, 12288, 3072, 32, name="flux_mlp_down_m4608_int4"),
        _case("linear", "nvfp4", 4608, 3072, 12288, 32, name="flux_mlp_up_m4608_nvfp4"),
        # the projection form with both kinds of operands; a picture whose token count fits no tile
        _case("linear", "int4_ph", 4173, 3072, 12288, 32, name="flux_mlp_up_m4173_int4_ph"),
        _case("linear", "nvfp4_ph", 4608, 12288, 3072, 32, name="flux_mlp_down_m4608_nvfp4_ph"),
        # a batch of four pictures, groups of 128
        _case("linear", "int4", 18432, 3072, 9216, 128, 128, name="flux_qkv_m18432_int4_g128"),
        # end to end from pinned host memory
        _case("host", "int4", 4608, 3072, 3072, 32, name="flux_out_m4608_host_int4"),
        # loading a layer
        _case("prepare", "int4", 1, 1152, 4608, 32, name="pixart_mlp_up_prepare_int4"),
    ]


def _log(rng, lo, hi, step=1):
    return max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)) * step)


def draw(rng):
    most = max(work(c)["flops"] for c in listed())
    while True:
        call = rng.choices(("linear", "shared", "host", "prepare"), (80, 8, 6, 6))[0]
        fmt = rng.choice(FORMATS) if call == "linear" else rng.choice(("int4", "int4_asym")) if call == "shared" else \
            rng.choice(("int4", "nvfp4_ph")) if call == "host" else "int4"
        M = 1 if call == "prepare" else _log(rng, 16, 18432)
        K, N = _log(rng, 512, 12288, 128), _log(rng, 512, 12288, 16)
        r = rng.choice((16, 32, 64, 128, max(16, round(0.1 * K / 16) * 16)))
        c = _case(call, fmt, M, K, N, r, rng.choice((64, 64, 128)))
        if work(c)["flops"] <= most:
            return c


def _rotation(K, r, outliers, basis, g):
    """Orthogonal [K, K] in fp64: the first r columns span the outlier channels, then the low-rank basis."""
    lead = torch.zeros((K, r), dtype=torch.float64, device="cuda")
    n_out = min(r, outliers.numel())
    lead[outliers[:n_out], torch.arange(n_out, device="cuda")] = 1.0
    n_basis = min(r - n_out, basis.shape[0])
    lead[:, n_out:n_out + n_basis] = basis[:n_basis].double().T
    lead[:, n_out + n_basis:] = torch.randn((K, r - n_out - n_basis), dtype=torch.float64, device="cuda", generator=g)
    a, tau = torch.geqrf(lead)
    Q = torch.ormqr(a, tau, torch.eye(K, dtype=torch.float64, device="cuda"))
    v = torch.randn(K - r, dtype=torch.float64, device="cuda", generator=g)
    v /= v.norm()
    low = Q[:, r:]
    low.sub_(torch.outer(low @ v, 2.0 * v))  # mixes the residual coefficients with one another
    return Q.contiguous()


class _State:
    pass


def prepare(case, seed):
    call, fmt, M, K, N, r, G = (case[k] for k in ("call", "fmt", "M", "K", "N", "r", "G"))
    g = torch.Generator(device="cuda").manual_seed(seed)
    model = synth.FLUX if K % 3072 == 0 else synth.PIXART
    outliers = torch.randperm(K, device="cuda", generator=g)[:model.n_outliers]
    gain = torch.ones(K, device="cuda")
    gain[outliers] = model.gain
    basis = torch.randn((model.rho, K), device="cuda", generator=g)
    x = torch.randn((M, K), device="cuda", generator=g) * gain
    x += (3.0 / math.sqrt(model.rho)) * (torch.randn((M, model.rho), device="cuda", generator=g) @ basis)
    x = x.to(torch.bfloat16)
    Q = _rotation(K, r, outliers, basis, g)
    bias = (0.02 * torch.randn(N, device="cuda", generator=g)).to(torch.bfloat16)

    def weight():
        return 0.02 * torch.randn((K, N), device="cuda", generator=g)

    s = _State()
    s.call, s.M = call, M
    if call == "prepare":
        s.W, s.Q, s.bias, s.r, s.G = weight(), Q, bias, r, G
        return s
    if fmt == "int4":
        s.layer = dq.dirotq_prepare_layer(weight(), Q, r, G, bias=bias)
    elif fmt == "int4_asym":
        s.layer = dq.dirotq_prepare_layer_asym(weight(), Q, r, G, bias=bias)
    elif fmt == "w4a8":
        s.layer = dq.dirotq_prepare_layer_w4a8(weight(), Q, r, bias=bias)
    elif fmt == "nvfp4":  # the activations' power-of-two scale is a calibration constant
        rotated = x[:1024].float() @ Q.float()
        s.layer = dq.dirotq_prepare_layer_nvfp4(weight(), Q, r, dq.dirotq_act_scale_log2_from_rotated(rotated, r), bias=bias)
    elif fmt == "int4_ph":
        s.layer = dq.dirotq_prepare_layer_ph(weight(), Q[:, :r].contiguous(), G, bias=bias)
    else:
        Uh = Q[:, :r].contiguous()
        s.layer = dq.dirotq_prepare_layer_nvfp4_ph(weight(), Uh, dq.dirotq_act_scale_log2_ph(x[:1024].contiguous(), Uh), bias=bias)
    s.ws = dq.alloc_workspace(s.layer, M)
    s.x = x
    s.y = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    if call == "shared":
        s.siblings = [dq.dirotq_prepare_layer_sibling(weight(), Q, r, G, bias=bias, asym=fmt == "int4_asym") for _ in range(2)]
        s.ys = [torch.empty_like(s.y) for _ in s.siblings]
    elif call == "host":
        s.x_host = torch.empty((M, K), dtype=torch.bfloat16, pin_memory=True)
        s.x_host.copy_(x)
        s.y_host = torch.empty((M, N), dtype=torch.bfloat16, pin_memory=True)
    return s


def run(s):
    if s.call == "linear":
        dq.dirotq_linear(s.x, s.layer, s.y, s.ws)
        return s.y
    if s.call == "shared":
        dq.dirotq_rotate_quantize(s.x, s.layer, s.ws)
        dq.dirotq_w4a4_gemm(s.M, s.layer, s.ws, s.y)
        for layer, y in zip(s.siblings, s.ys):
            dq.dirotq_w4a4_gemm(s.M, layer, s.ws, y)
        return [s.y, *s.ys]
    if s.call == "host":
        dq.dirotq_linear_host(s.x_host, s.layer, s.y_host, s.x, s.y, s.ws)
        return s.y_host
    layer = dq.dirotq_prepare_layer(s.W, s.Q, s.r, s.G, bias=s.bias)
    codes, scales, high, rotation = dq.dirotq_layer_export(layer)
    layer.close()
    return [codes, scales, high, rotation]


def work(case):
    call, fmt, M, K, N, r, G = (case[k] for k in ("call", "fmt", "M", "K", "N", "r", "G"))
    if call == "prepare":
        groups = -(-(K - r) // G)
        made = (K - r) * N + 2 * groups * N + 2 * r * N + 2 * K * K  # codes, scales, 16-bit rows, rotation: exported one byte per code
        return {"bytes": 4 * K * N + 8 * K * K + 2 * N + made, "flops": 2.0 * K * K * N}
    ph = fmt.endswith("_ph")
    low = K if ph else K - r
    layers = 3 if call == "shared" else 1
    scales = 2 * N if fmt == "w4a8" else low / 16 * N if fmt.startswith("nvfp4") else 2 * -(-low // G) * N
    first_bytes = 4 * r * K if ph else 2 * K * K
    first_flops = 4.0 * M * K * r + 2.0 * M * K * (64 if fmt == "nvfp4_ph" else G) if ph else 2.0 * M * K * K
    return {"bytes": 2 * M * K + first_bytes + layers * (low * N / 2 + scales + 2 * r * N + 2 * N + 2 * M * N),
            "flops": first_flops + layers * 2.0 * M * K * N}


def tolerance(case):
    if case["call"] == "prepare":  # folded in fp64: codes differ only where a quotient is a tie to within fp64 rounding
        return {"rel": 1e-4, "max": 0.01, "differ": 1e-6}
    # bf16 results; a rotated coefficient that lies on a rounding boundary may take the neighbouring code
    return {"rel": 1e-2, "max": 0.1}

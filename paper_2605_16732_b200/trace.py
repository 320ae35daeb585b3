"""Clock traces of the kernels' roles, read off the device.

    python -m paper_2605_16732_b200.trace [--what small_m | w4a4 | nvfp4 | w4a8 | w4a8_single]

Builds the diagnostic library (`build.build_trace()`: the same sources with -DDIROTQ_TRACE, in which block 0 of every kernel stamps
`clock64()` at marked points of its roles into spare 8-byte slots of the workspace's status block), runs one workload on it and
prints the stamps as cycles since the kernel's entry.  The slot map is documented at each kernel's first stamp; the plans are
forced, so that the kernel a title names is the one that ran, and a stamp that is missing is an error.

    small_m      the small layer (M = 256, 1152 -> 1152, r = 32, groups of 64), each INT4 kernel replayed alone from a CUDA graph
    w4a4         the INT4 second kernel, 256-column tiles, on the FLUX qkv shape (M = 4608, 3072 -> 9216)
    nvfp4        the second kernel of the NVFP4 format (CTA pairs) behind the projection form on the same shape
    w4a8         the second kernel of the W4A8 format in CTA pairs, 256-column tiles, on the same shape
    w4a8_single  its single-CTA form (128-column tiles) on the same shape
"""
from __future__ import annotations

import argparse
import sys

# Per kernel: the slot of its entry stamp, and what the others mean, in the order they are printed.
W4A4_SLOTS = (9, [("set-up done / previous grid ended", (10, 11)), ("producer: first k-block issued / everything issued", (12, 13)),
                  ("first unpack warp: first stage seen / expanded", (14, 15)),
                  ("MMA warp: first / fifth / last k-block, last tile committed", (16, 17, 18, 19)),
                  ("first epilogue warp: first accumulator / ninth group / groups done / rank-r done / stored", (20, 21, 22, 23, 24))])
SLOTS = {
    "rotate_quant_kernel": (9, [("set-up done / previous grid ended", (10, 11)), ("producer: ring filled once / everything issued", (12, 13)),
                                ("MMA warp: first / ninth stage seen, last tile committed", (14, 15, 16)),
                                ("first epilogue warp: first accumulator seen / finished", (17, 18))]),
    "w4a4_narrow_kernel": W4A4_SLOTS,
    "w4a4_gemm_kernel": W4A4_SLOTS,  # (the last tile's stamps where a CTA has several)
    "nvfp4_gemm_kernel": (30, [("stages 6, 7, 8 of the first tile: producer has issued the stage", (9, 10, 11)),
                               ("first copier warp sees it landed", (12, 13, 14)), ("first copier warp committed", (15, 16, 17)),
                               ("second copier warp committed", (18, 19, 20)), ("MMA warp sees the scales ready", (21, 22, 23)),
                               ("MMA warp committed the stage", (24, 25, 26)),
                               ("epilogue tile 0: accumulator seen / released / handed over", (27, 28, 29)),
                               ("epilogue tile 1", (1, 2, 3)), ("epilogue tile 2", (4, 5, 6))]),
    "w4a8_pair_kernel": (30, [("previous grid ended", (31,)), ("k-blocks 18, 19, 20 of the first tile: packed weights issued", (9, 10, 11)),
                              ("an expanding team sees them landed", (12, 13, 14)), ("it has an operand slot", (15, 16, 17)),
                              ("it has expanded them", (18, 19, 20)), ("MMA warp sees the k-block", (21, 22, 23)),
                              ("MMA warp has issued it", (24, 25, 26))]),
    "w4a8_gemm_kernel": (30, [("stages 10, 11, 12 of the first tile: producer has issued the stage", (9, 10, 11)),
                              ("first unpack warp sees it landed", (12, 13, 14)), ("first unpack warp has expanded it", (15, 16, 17)),
                              ("MMA warp starts on it", (18, 19, 20)), ("epilogue tile 0: accumulators seen / released / handed over", (21, 22, 23)),
                              ("epilogue tile 1", (24, 25, 26)), ("epilogue tile 2", (27, 28, 29))]),
}
# second kernels on the FLUX qkv shape: format, kernel, the tile plan that names it (dirotq_set_gemm_tile)
WIDE = {"w4a4": ("int4", "w4a4_gemm_kernel", 256), "nvfp4": ("nvfp4_ph", "nvfp4_gemm_kernel", 512),
        "w4a8": ("w4a8", "w4a8_pair_kernel", 512), "w4a8_single": ("w4a8", "w4a8_gemm_kernel", 128)}


def _show(kernel, note, ws):
    import torch
    torch.cuda.synchronize()
    st = ws[:256].view(torch.int64).cpu().tolist()
    entry, names = SLOTS[kernel]
    print(f"{kernel}, {note}; cycles since entry of block 0")
    for name, slots in names:
        for i in slots:
            if not 0 < st[entry] <= st[i]:
                raise RuntimeError(f"{kernel}: no stamp in slot {i} ({name})")
        print("   %-92s %s" % (name, " ".join(str(st[i] - st[entry]) for i in slots)))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--what", default="small_m", choices=["small_m", *WIDE])
    args = ap.parse_args()
    from . import binding as dq, build
    dq.use_library(build.build_trace())  # before the binding loads a library
    from . import suite, synth

    if args.what == "small_m":
        c = suite.Case(256, 1152, 1152, 32, 64, synth.PIXART)
        dq.dirotq_set_rotation_tile(5)
        dq.dirotq_set_gemm_tile(32)
        us = c.graph_ms(lambda: dq.dirotq_rotate_quantize(c.x, c.layer, c.ws)) * 1e3
        _show("rotate_quant_kernel", f"128 x 64 tiles, {us:.2f} us per call in graph replay", c.ws)
        c.ws[:256].zero_()
        us = c.graph_ms(lambda: dq.dirotq_w4a4_gemm(c.M, c.layer, c.ws, c.y)) * 1e3
        _show("w4a4_narrow_kernel", f"128 x 32 tiles, {us:.2f} us per call in graph replay", c.ws)
    else:
        suite.FMT, kernel, tile = WIDE[args.what]
        c = suite.Case(4608, 3072, 9216, 32, 64, synth.FLUX)
        dq.dirotq_set_gemm_tile(tile)
        dq.dirotq_rotate_quantize(c.x, c.layer, c.ws)
        c.ws[:256].zero_()
        for _ in range(3):
            dq.dirotq_w4a4_gemm(c.M, c.layer, c.ws, c.y)
        _show(kernel, "FLUX qkv", c.ws)
    assert dq.dirotq_workspace_status(c.ws) == 0
    c.close()


if __name__ == "__main__":
    sys.exit(main())

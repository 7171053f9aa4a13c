"""The work that users of the library have it do, as measurable cases.

A case describes one 3x3 stride-1 layer (or a short chain of them) and the entry point it
goes through:

* ``op = "forward"``       ``Conv.forward`` on CUDA tensors, `depth` layers one after another
* ``op = "forward_host"``  ``Conv.forward_host`` on pinned host tensors, copies included
* ``op = "prepare"``       ``Conv.prepare``: filter transform and quantization when weights arrive

Shapes and value distributions are those of the benchmark configurations (ResNet-18/34 stages,
diffusion-UNet conv blocks) and of the tests.
"""
import math

import torch

from paper_2412_19867_b200 import binding, workloads

DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
ACTS = {"none": binding.WFQ_ACT_NONE, "relu": binding.WFQ_ACT_RELU, "silu": binding.WFQ_ACT_SILU}


def _case(N, C, K, H, W, m, gs, op="forward", depth=1, dtype="f16", layout="nchw", out="f32", act="none",
          bias=False, values="relu_heavy", quant="none", w_bits=8):
    return dict(op=op, depth=depth, N=N, C=C, K=K, H=H, W=W, m=m, gs=gs, dtype=dtype, layout=layout, out=out,
                act=act, bias=bias, values=values, quant=quant, w_bits=w_bits)


def listed():
    silu = dict(values="silu_outlier")
    named = {
        # one small fp32 image through one layer: latency of a single call
        "single_32x32_f32": _case(1, 64, 64, 32, 32, 4, 32, dtype="f32", values="gauss_outlier"),
        # first ResNet-18 stage, batch 32: many tiles, few channels, fp32 result for the caller's own code
        "resnet_56x56": _case(32, 64, 64, 56, 56, 6, 64),
        # a ResNet basic block of the last stage (two layers, folded batch norm, ReLU, fp16 in between):
        # odd 7x7 images that fill the second tile of a row with one column
        "resnet_block_7x7": _case(32, 512, 512, 7, 7, 6, 64, depth=2, out="f16", act="relu", bias=True),
        # ResNet-34 stage, batch 64, the smaller tile and the smallest groups; ragged 14 = 3 * 4 + 2
        "resnet_14x14_g32": _case(64, 256, 256, 14, 14, 4, 32),
        # ResNet-34 stage, batch 64, in a channels-last network with groups of 128
        "resnet_28x28_nhwc": _case(64, 128, 128, 28, 28, 6, 128, layout="nhwc", out="f16", act="relu", bias=True),
        # the UNet's highest resolution, one image
        "unet_128x128": _case(1, 320, 320, 128, 128, 4, 64, **silu),
        # a UNet residual block (two layers with SiLU) in classifier-free guidance (two images)
        "unet_block_32x32": _case(2, 640, 640, 32, 32, 4, 64, depth=2, out="f16", act="silu", bias=True, **silu),
        # the UNet's widest layer: 105 MB of filter codes against 1.3 million input values
        "unet_1280_32x32": _case(1, 1280, 1280, 32, 32, 6, 64, **silu),
        # a UNet layer in a channels-last pipeline with bf16 results
        "unet_64x64_nhwc": _case(1, 640, 640, 64, 64, 6, 64, layout="nhwc", out="bf16", act="silu", bias=True, **silu),
        # the paper's fully quantized setting: integer input and output transforms, one scale per tile
        "unet_32x32_fullquant": _case(2, 640, 640, 32, 32, 4, 64, quant="tile", **silu),
        # loading a layer's weights into a plan
        "filters_640x1280": _case(1, 640, 1280, 32, 32, 6, 64, op="prepare", **silu),
        # a batch that lives in pinned host memory, fp16 both ways
        "host_28x28": _case(32, 128, 128, 28, 28, 6, 64, op="forward_host", out="f16"),
    }
    return [dict(name=name, **case) for name, case in named.items()]


def _effort(case):
    """Rough cost of a pass in bytes moved, to keep drawn cases within the listed ones of their kind."""
    total = 0.0
    for C, K in _layers(case):
        P, T = (case["m"] + 2) ** 2, (0 if case["op"] == "prepare" else _tiles(case))
        total += P * C * K + P * T * (2.0 * C + 8.0 * K) + P * T * C * K / 500.0
    return total * (2.0 if case["quant"] != "none" else 1.0)


def draw(rng):
    limit = {}
    for c in listed():
        limit[c["op"]] = max(limit.get(c["op"], 0.0), _effort(c))

    def spread(lo, hi, step=1):
        return max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.5 * step))) / step)) * step)

    while True:
        gs = rng.choice([32, 64, 64, 128])
        C = spread(gs, 1280, gs)
        K = rng.choice([C, spread(16, 1280, 8)])
        H = spread(5, 136)
        W = rng.choice([H, H, spread(5, 136)])
        N = spread(1, 64)
        m = rng.choice([4, 4, 4, 6, 6, 6, 2])
        op = rng.choice(["forward"] * 8 + ["forward_host", "prepare"])
        dtype = rng.choice(["f16"] * 6 + ["f32"])
        layout = rng.choice(["nchw", "nchw", "nhwc"])
        depth = 1
        out, act, bias = rng.choice([("f32", "none", False), ("f16", "relu", True), ("f16", "silu", True),
                                     ("bf16", "none", True)])
        quant = "none"
        if op == "forward" and layout == "nchw":
            kind = rng.randrange(8)
            if kind == 0:
                quant = rng.choice(["tile", "row"])
            elif kind <= 2 and K % gs == 0 and dtype == "f16":
                depth, out = 2, "f16"
        values = rng.choice(["relu_heavy", "silu_outlier", "gauss_outlier"])
        w_bits = rng.choice([8] * 7 + [4])
        case = _case(N, C, K, H, W, m, gs, op=op, depth=depth, dtype=dtype, layout=layout, out=out, act=act,
                     bias=bias, values=values, quant=quant, w_bits=w_bits)
        if _effort(case) <= limit[op]:
            return case


def _layers(case):
    """(input channels, output channels) of the chain's layers."""
    return [(case["C"] if i == 0 else case["K"], case["K"]) for i in range(case["depth"])]


def _tiles(case):
    return case["N"] * -(-case["H"] // case["m"]) * -(-case["W"] // case["m"])


def _activations(gen, case):
    shape = (case["N"], case["C"], case["H"], case["W"])
    if case["layout"] == "nhwc":
        shape = (case["N"], case["H"], case["W"], case["C"])
    z = torch.randn(shape, generator=gen, device="cuda")
    if case["values"] == "relu_heavy":
        # relu of a Student-t(4): chi-square(4) = -2 log(u1 u2)
        u = torch.rand((2,) + shape, generator=gen, device="cuda").clamp_(min=1e-7)
        x = (z / torch.sqrt(-0.5 * torch.log(u[0] * u[1]))).clamp_(min=0.0)
    elif case["values"] == "silu_outlier":
        x = z * torch.sigmoid(z)
        x = torch.where(torch.rand(shape, generator=gen, device="cuda") < 0.005, 50.0 * x, x)
    else:
        x = torch.where(torch.rand(shape, generator=gen, device="cuda") < 0.01, 20.0 * z, z)
    return x.to(DTYPES[case["dtype"]]).contiguous()


def _filters(gen, case, C, K):
    w = torch.randn((K, C, 3, 3), generator=gen, device="cuda") * math.sqrt(2.0 / (9 * C))
    if case["values"] != "relu_heavy":        # output channels of very different sizes
        u = torch.rand((K, 1, 1, 1), generator=gen, device="cuda")
        w = w * torch.exp(math.log(0.1) + u * (math.log(10.0) - math.log(0.1)))
    return w.contiguous()


def _scales(gen, m):
    def vector(std):
        z = torch.randn(len(std), generator=gen, device="cuda").tolist()
        return [s * math.exp(0.1 * v) for s, v in zip(std, z)]
    return vector(workloads.STD_SB[m]), vector(workloads.STD_SG[m])


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = _activations(gen, case) if case["op"] != "prepare" else None
    layers = []
    for i, (C, K) in enumerate(_layers(case)):
        w = _filters(gen, case, C, K)
        sB, sG = _scales(gen, case["m"])
        conv = binding.Conv(case["N"], C, K, case["H"], case["W"], case["m"], case["gs"],
                            case["dtype"] if i == 0 else case["out"])
        if i == 0 and case["layout"] == "nhwc":
            conv.set_input_layout("nhwc")
        conv.set_weight_bits(case["w_bits"])
        conv.set_output_dtype(case["out"])
        if case["quant"] != "none":
            binding.wfq_plan_set_full_quant(conv.plan, 1,
                                            binding.WFQ_Y_TILE if case["quant"] == "tile" else binding.WFQ_Y_ROW)
        bias = 0.1 * torch.randn(K, generator=gen, device="cuda") if case["bias"] else None
        conv.set_epilogue(bias, ACTS[case["act"]])
        if case["op"] != "prepare":
            conv.prepare(w, sB, sG)
        layers.append((conv, w, sB, sG))
    state = {"op": case["op"], "layers": layers, "x": x}
    if case["op"] == "forward_host":
        state["x"] = torch.empty(x.shape, dtype=x.dtype, pin_memory=True).copy_(x)
        state["y"] = torch.empty((case["N"], case["K"], case["H"], case["W"]), dtype=DTYPES[case["out"]],
                                 pin_memory=True)
    return state


def run(state):
    if state["op"] == "prepare":
        conv, w, sB, sG = state["layers"][0]
        conv.prepare(w, sB, sG)
        out = {"codes": conv.buffer(binding.WFQ_BUF_WQ), "scales": conv.buffer(binding.WFQ_BUF_SW)}
        for tensor in out.values():
            tensor.owner = conv          # views of the plan's memory: the plan has to outlive them
        return out
    if state["op"] == "forward_host":
        return state["layers"][0][0].forward_host(state["x"], state["y"])
    x = state["x"]
    for conv, _, _, _ in state["layers"]:
        x = conv.forward(x)
    return x


def work(case):
    esz = {"f32": 4, "f16": 2, "bf16": 2}
    pixels = case["N"] * case["H"] * case["W"]
    P, T = (case["m"] + 2) ** 2, _tiles(case)
    nbytes = flops = 0.0
    for i, (C, K) in enumerate(_layers(case)):
        filters = P * K * C + 4.0 * P * (C // case["gs"]) * K        # codes and group scales
        if case["op"] == "prepare":
            n = case["m"] + 2
            nbytes += 4.0 * 9 * K * C + filters
            flops += K * C * 2.0 * (9 * n + 3 * n * n)               # V_G w V_G^T
        else:
            nbytes += pixels * C * esz[case["dtype"] if i == 0 else case["out"]] + filters
            nbytes += pixels * K * esz[case["out"]]
            flops += 2.0 * P * T * C * K                             # the contraction
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Measured against the same pipeline with its transforms and sums in 64 bits (the CPU oracle) on
    these cases and forty drawn ones.  What shows is not the 32-bit arithmetic (1e-6 where no code
    differs) but a value within rounding of the middle between two int8 codes: one step of a group that
    holds an outlier moves m x m outputs of one tile."""
    if case["op"] == "prepare":
        # 64-bit arithmetic rounded once to 32 bits: another order of the sums changes next to nothing
        return {"rel": 1e-6, "differ": 1e-6}
    if case["quant"] != "none":
        # every quantizer decides in 64 bits, on a contraction result in 32 bits: a relative error of
        # 3e-7 there moves about 2e-5 of its codes by one step in (typically) 30
        return {"rel": 1e-3}
    # one layer: 7e-4 at most.  A second layer quantizes the 16-bit results of the first, of which those
    # that a code of the first moved differ: 3.9e-3 at most.
    return {"rel": 3e-3 if case["depth"] == 1 else 1.6e-2}

"""The calls that this library is used for, as cases that can be timed and compared.

A case is one pass of a program that uses the module: a super-resolution forward on one feature map, the module with its
closing 1x1 convolution, a backward pass on a batch of training patches, a call on host buffers.  The sizes are the ESC
networks' (LR maps of 320x180, 427x240 and 640x360 for a 1280x720 result, training batches of 64x64 patches, widths 64, 48
and 192) and this repository's own workloads.

Keys of a case: op ("forward_fixed": the fp32 NCHW entry with library-owned scratch; "forward"; "module": forward, Conv_fuse
and residual in one call; "backward": Conv_fuse's backward, then the module's; "host": host buffers in and out), form of the
large kernel ("depthwise", "decomposed", "dense"), hidden (0: one linear layer as kernel estimator, else the width of the
two-layer one), dtype, layout, and the sizes B, C, C_a, H, W, K.
"""
import math

import torch

import paper_2503_06671_b200 as esc

FORMS = {"depthwise": esc.ESC_LK_DEPTHWISE, "decomposed": esc.ESC_LK_DECOMPOSED, "dense": esc.ESC_LK_DENSE}
DTYPES = {"fp32": torch.float32, "bf16": torch.bfloat16}
LAYOUTS = {"nchw": esc.ESC_NCHW, "nhwc": esc.ESC_NHWC}


def _case(name, op, form, hidden, dtype, layout, B, C, C_a, H, W, K=13):
    return {"name": name, "op": op, "form": form, "hidden": hidden, "dtype": dtype, "layout": layout,
            "B": B, "C": C, "C_a": C_a, "H": H, "W": W, "K": K}


def listed():
    return [
        # one small fp32 map: latency of a single call (a preview, an interactive crop)
        _case("crop_fp32_64x64", "forward_fixed", "depthwise", 0, "fp32", "nchw", 1, 64, 16, 64, 64),
        # LR map of x4 super-resolution to 1280x720 in the paper's precision
        _case("x4_fp32_320x180", "forward_fixed", "depthwise", 0, "fp32", "nchw", 1, 64, 16, 180, 320),
        # LR map of x2 super-resolution, mixed precision, channels last: the module of the benchmark
        _case("x2_bf16_nhwc_640x360", "forward", "depthwise", 0, "bf16", "nhwc", 1, 64, 16, 360, 640),
        # the largest map: x2 to 4K with 32 attention channels
        _case("uhd_bf16_nhwc_1920x1080", "forward", "depthwise", 0, "bf16", "nhwc", 1, 64, 32, 1080, 1920),
        # ESC (dense large kernel, two-layer estimator), x2, mixed precision
        _case("esc_x2_bf16_nhwc_640x360", "forward", "dense", 8, "bf16", "nhwc", 1, 64, 16, 360, 640),
        # the same network in fp32 and PyTorch's default layout: the configuration the paper times
        _case("esc_x2_fp32_nchw_640x360", "forward", "dense", 8, "fp32", "nchw", 1, 64, 16, 360, 640),
        # ESC-FP (decomposed large kernel, 48 channels), x3: the LR map has an odd width
        _case("escfp_x3_bf16_nchw_427x240", "forward", "decomposed", 8, "bf16", "nchw", 1, 48, 16, 240, 427),
        # the whole module in one call: forward, closing 1x1 convolution and the block's residual
        _case("module_x2_bf16_nhwc_640x360", "module", "depthwise", 0, "bf16", "nhwc", 1, 64, 16, 360, 640),
        # training ESC: a batch of 64 patches, channels last, backward of the module and of its 1x1 convolution
        _case("train_esc_bf16_nhwc_64x64x64", "backward", "dense", 8, "bf16", "nhwc", 64, 64, 16, 64, 64),
        # training ESC-FP in PyTorch's default layout
        _case("train_escfp_bf16_nchw_32x64x64", "backward", "decomposed", 4, "bf16", "nchw", 32, 48, 16, 64, 64),
        # training in fp32 (depth-wise kernel), a small batch as for fine-tuning
        _case("train_fp32_nchw_8x64x64", "backward", "depthwise", 0, "fp32", "nchw", 8, 64, 16, 64, 64),
        # host buffers in, host buffers out, one blocking call
        _case("host_bf16_nhwc_640x360", "host", "depthwise", 0, "bf16", "nhwc", 1, 64, 16, 360, 640),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _map_size(rng, most):
    """Height and width of a feature map of at most `most` pixels: any aspect a picture has, odd sizes as well as round ones."""
    H = _log_int(rng, 48, math.sqrt(most * 9 / 16))
    W = min(int(H * rng.choice([1.0, 4 / 3, 1.5, 16 / 9])), most // H)
    if rng.random() < 0.6:
        H, W = max(48, H // 8 * 8), max(48, W // 8 * 8)
    return H, W


def draw(rng):
    dtype = rng.choice(["bf16", "bf16", "fp32"])
    layout = rng.choice(["nhwc", "nchw"])
    op = rng.choice(["forward", "forward", "forward", "module", "backward", "backward", "host"])
    form = "depthwise" if op in ("module", "host") else rng.choice(["depthwise", "decomposed", "dense"])
    hidden = 0 if op in ("module", "host") else rng.choice([0, 4, 8])
    C, C_a = rng.choice([(64, 16), (64, 16), (48, 16)])
    if op == "forward" and form == "depthwise":
        C, C_a = rng.choice([(64, 16), (48, 16), (64, 32), (192, 48)])
    K = rng.choice([13, 13, 13, 13, 9])
    if op == "forward" and form == "depthwise" and rng.random() < 0.1:
        K = 17
    if op == "backward" or (op == "forward" and rng.random() < 0.25):
        B = _log_int(rng, 4, 64)                             # a batch of training patches
        H = W = rng.choice([48, 64, 64, 96]) if rng.random() < 0.7 else rng.randrange(41, 97)
        most = 64 if (dtype, layout) == ("bf16", "nhwc") else 40
        B = min(B, most * 64 * 64 // (H * W))
    else:
        B = 1
        most = 1920 * 1080 if form == "depthwise" and dtype == "bf16" and op == "forward" and C == 64 else 640 * 360
        H, W = _map_size(rng, most)
    c = _case("", op, form, hidden, dtype, layout, B, C, C_a, H, W, K)
    del c["name"]
    return c


def _weights(case, g):
    C, C_a, K, h = case["C"], case["C_a"], case["K"], case["hidden"]

    def uniform(*shape, fan_in):
        bound = 1.0 / math.sqrt(fan_in)
        return (torch.rand(*shape, generator=g, device="cuda") * (2 * bound) - bound).to(DTYPES[case["dtype"]])

    w = {}
    w["large"] = uniform(C_a, C_a, K, K, fan_in=C_a * K * K) if case["form"] == "dense" else uniform(C_a, K, K, fan_in=K * K)
    w["point"] = uniform(C_a, C_a, fan_in=C_a) if case["form"] == "decomposed" else None
    w["down"] = uniform(h, C_a, fan_in=C_a) if h else None
    w["b_down"] = uniform(h, fan_in=C_a) if h else None
    w["up"] = uniform(9 * C_a, h or C_a, fan_in=h or C_a)
    w["b_up"] = uniform(9 * C_a, fan_in=h or C_a)
    w["fuse"] = uniform(C, C, fan_in=C)
    w["b_fuse"] = uniform(C, fan_in=C)
    return w


def prepare(case, seed):
    """Inputs, weights, outputs and workspace: what a program holds before the call.  Activations have a mean per image and
    channel and a scale per image, as feature maps do; without them the global average pool would have nothing to say."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    B, C, C_a, H, W, K = (case[k] for k in ("B", "C", "C_a", "H", "W", "K"))
    nhwc = case["layout"] == "nhwc"
    shape = (B, H, W, C) if nhwc else (B, C, H, W)
    per_channel = (B, 1, 1, C) if nhwc else (B, C, 1, 1)
    dt = DTYPES[case["dtype"]]

    def activations():
        t = torch.randn(shape, generator=g, device="cuda")
        t *= torch.rand((B, 1, 1, 1), generator=g, device="cuda") + 0.5
        t += torch.randn(per_channel, generator=g, device="cuda") * 0.5
        return t.to(dt)

    s = {"case": dict(case), "layout": LAYOUTS[case["layout"]], "x": activations(), "w": _weights(case, g)}
    op = case["op"]
    if op == "host":
        s["x"] = s["x"].cpu().pin_memory()
        s["w"] = {k: v.cpu().pin_memory() for k, v in s["w"].items() if v is not None}
        s["out"] = torch.empty_like(s["x"], pin_memory=True)
    elif op == "backward":
        # the concatenated map in front of the 1x1 convolution: the identity channels are x's own
        att = activations()
        a, i = ([att[..., :C_a], s["x"][..., C_a:]] if nhwc else [att[:, :C_a], s["x"][:, C_a:]])
        s["cat"] = torch.cat([a, i], dim=3 if nhwc else 1).contiguous()
        s["go"] = torch.randn(shape, generator=g, device="cuda").to(dt)
        s["g_cat"], s["g_x"] = torch.empty_like(s["x"]), torch.empty_like(s["x"])
        s["g"] = {k: torch.zeros(v.shape, device="cuda") for k, v in s["w"].items() if v is not None}
        dense = case["form"] == "dense"
        s["ws"] = (esc.new_backward_dense_workspace if dense else esc.new_backward_workspace)(B, C_a, H, W, K)
        n = esc.esc_conv_fuse_backward_workspace_bytes(B, C, H, W)
        s["ws_fuse"] = torch.empty(n, dtype=torch.uint8, device="cuda")
    else:
        s["out"] = torch.empty_like(s["x"])
        if op == "module":
            s["residual"] = activations()
        if op != "forward_fixed":
            s["ws"] = esc.new_workspace(B, C_a, H, W, K)
    return s


def run(s):
    case, w, layout = s["case"], s["w"], s["layout"]
    op, C_a, K = case["op"], case["C_a"], case["K"]
    if op == "forward_fixed":
        return esc.esc_convattn_forward(s["x"], C_a, K, w["large"], w["up"], w["b_up"], s["out"])
    if op == "forward":
        if case["form"] == "depthwise" and not case["hidden"]:
            return esc.esc_convattn_forward_ex(s["x"], C_a, K, w["large"], w["up"], w["b_up"], s["out"], layout, s["ws"])
        return esc.esc_convattn_forward_variant(s["x"], C_a, K, FORMS[case["form"]], w["large"], w["point"], w["down"], w["b_down"],
                                                w["up"], w["b_up"], s["out"], layout, s["ws"])
    if op == "module":
        return esc.esc_convattn_forward_fused(s["x"], C_a, K, w["large"], w["up"], w["b_up"], w["fuse"], w["b_fuse"], s["residual"],
                                              s["out"], layout, s["ws"])
    if op == "host":
        return esc.esc_convattn_forward_host(s["x"], C_a, K, w["large"], w["up"], w["b_up"], s["out"], layout)
    g = s["g"]
    esc.esc_conv_fuse_backward(s["cat"], s["go"], w["fuse"], s["g_cat"], g["fuse"], g["b_fuse"], layout, s["ws_fuse"])
    if case["form"] == "depthwise" and not case["hidden"]:
        esc.esc_convattn_backward(s["x"], s["g_cat"], C_a, K, w["large"], w["up"], w["b_up"], s["g_x"], g["large"], g["up"],
                                  g["b_up"], layout, s["ws"])
    else:
        esc.esc_convattn_backward_variant(s["x"], s["g_cat"], C_a, K, FORMS[case["form"]], w["large"], w["point"], w["down"],
                                          w["b_down"], w["up"], w["b_up"], s["g_x"], g["large"], g.get("point"), g.get("down"),
                                          g.get("b_down"), g["up"], g["b_up"], layout, s["ws"])
    return {"g_x": s["g_x"], "g_cat": s["g_cat"], **{"g_" + k: v for k, v in g.items()}}


def work(case):
    """Each tensor of each call read or written once; multiply-adds of the convolutions, counted as two operations.  The
    backward pass is two calls: the first reads cat and grad_out and writes g_cat, the second reads g_cat and the attention
    channels of x and writes g_x; every convolution costs its forward's operations twice."""
    B, C, C_a, H, W, K = (case[k] for k in ("B", "C", "C_a", "H", "W", "K"))
    px = B * H * W
    es = 4 if case["dtype"] == "fp32" else 2
    form, op = case["form"], case["op"]
    macs = px * C_a * ((C_a * K * K + 9) if form == "dense" else K * K)
    if form == "decomposed":
        macs += px * C_a * C_a
    if op in ("module", "backward"):
        macs += px * C * C
    maps = {"module": 3, "backward": 5 + C_a / C}.get(op, 2)
    return {"bytes": int(maps * px * C * es), "flops": 2 * macs * (2 if op == "backward" else 1)}


def tolerance(case):
    """Measured against the same passes in 64 bits, over these cases and drawn ones, and stated at about four times that.
    fp32: 5e-7 at most in the 2-norm, 6e-6 for one value.  bf16: 2.6e-3 and 1.1e-2 (one rounding of a result, another where
    the path stores an intermediate map)."""
    return {"rel": 2e-6, "max": 2.5e-5} if case["dtype"] == "fp32" else {"rel": 1e-2, "max": 4e-2}

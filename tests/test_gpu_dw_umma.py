"""The tcgen05 depth-wise kernel (bf16 NHWC, two or more groups of 16 channels, more work than the one-launch form takes) against the oracle: windows that hold many small
images, image rows of one to a few hundred pixels, row segments, channel groups, every kernel size's ends, the copied channels, the
constant per (image, channel) of the backward pass, and the reach of a non-finite input."""
import numpy as np
import pytest

from paper_2503_06671_b200 import synth
from tests import test_gpu_fuse, test_gpu_mlp, test_gpu_parity, util

pytestmark = pytest.mark.gpu

SHAPES = [
    # B, C, C_a, H, W, K: more than 1,184 tiles of 64x16 x 16 channels
    (700, 32, 32, 3, 1, 13),         # 38 images in a window, nothing to copy
    (150, 40, 32, 70, 7, 9),         # 20 images in a window, 8 channels copied
    (600, 64, 32, 5, 40, 13),        # images shorter than the kernel
    (600, 48, 32, 20, 33, 3),        # four octets, odd width
    (420, 64, 48, 9, 67, 11),        # six octets
    (2, 40, 32, 300, 1001, 13),      # windows that begin in one row segment and end in the next; rows copied one by one
    (1, 64, 32, 1213, 1030, 5),      # one image, a last window that is nearly empty
    (1, 192, 48, 420, 1000, 7),      # chunks of 32 pixels
]


@pytest.fixture(scope="module")
def pkg():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import paper_2503_06671_b200 as p

    p.lib()
    return p


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_stage_against_oracle(pkg, shape):
    import torch

    import oracle

    B, C, C_a, H, W, K = shape
    d = synth.make_inputs(B, C, C_a, H, W, K, synth.BF16, seed=sum(shape) + 1)
    dk = np.random.default_rng(6).uniform(-0.5, 0.5, size=(B, C_a, 3, 3)).astype(np.float32)
    x = util.to_device(d["x"], synth.BF16, synth.NHWC)
    wl, _, _ = util.weights_to_device(d, synth.BF16)
    n = x.numel()
    buf = torch.full((n + 4096,), 7.0, dtype=x.dtype, device="cuda")
    out = buf[2048:2048 + n].view(x.shape)
    ws = pkg.new_workspace(B, C_a, H, W, K)
    for _ in range(2):
        pkg.esc_convattn_stencil(x, C_a, K, wl, torch.from_numpy(dk).cuda(), out, pkg.ESC_NHWC, ws)
    torch.cuda.synchronize()
    assert pkg.esc_convattn_device_status(ws) == 0
    assert pkg.esc_convattn_last_path() == 4 and pkg.esc_convattn_last_tile_width() == 256
    assert bool((buf[:2048] == 7.0).all()) and bool((buf[2048 + n:] == 7.0).all()), "write outside out"
    ref, mag = oracle.stencil(d["x"], C_a, d["w_large"], dk, want_mag=True)
    got = util.to_host_nchw(out, synth.NHWC)
    util.check_attention(got[:, :C_a], ref[:, :C_a], mag, synth.BF16, f"{shape}", unit_variance=True)
    assert np.array_equal(got[:, C_a:], ref[:, C_a:])


@pytest.mark.parametrize("C_a, width", [(304, 256), (400, 64)])
def test_many_channels(pkg, oracle, C_a, width):
    """A group of CTAs takes one for every eight channels: where those groups leave more than a quarter of the 148 SMs empty (400
    channels: two of 50; 304: three of 38) the mma.sync kernel is the faster one and stays."""
    import torch

    B, H, W, K = 8, 100, 66, 5
    d = synth.make_inputs(B, C_a, C_a, H, W, K, synth.BF16, seed=C_a)
    dk = np.random.default_rng(6).uniform(-0.5, 0.5, size=(B, C_a, 3, 3)).astype(np.float32)
    x = util.to_device(d["x"], synth.BF16, synth.NHWC)
    wl, _, _ = util.weights_to_device(d, synth.BF16)
    out, ws = torch.empty_like(x), pkg.new_workspace(B, C_a, H, W, K)
    pkg.esc_convattn_stencil(x, C_a, K, wl, torch.from_numpy(dk).cuda(), out, pkg.ESC_NHWC, ws)
    torch.cuda.synchronize()
    assert pkg.esc_convattn_device_status(ws) == 0 and pkg.esc_convattn_last_tile_width() == width
    ref, mag = oracle.stencil(d["x"], C_a, d["w_large"], dk, want_mag=True)
    util.check_attention(util.to_host_nchw(out, synth.NHWC), ref, mag, synth.BF16, f"C_a = {C_a}", unit_variance=True)


@pytest.mark.parametrize("shape", [(64, 64, 32, 50, 130, 13), (1, 48, 32, 700, 901, 13), (64, 64, 32, 50, 130, 9), (1, 96, 48, 500, 800, 5), (80, 112, 96, 40, 40, 11)],
                         ids=lambda s: "x".join(map(str, s)))
def test_forward(pkg, oracle, shape):
    """Behind the pooling kernel and the linear estimator, as a programmatic dependent: batches and single images, K below 13, more than
    64 channels (a smaller pooling grid)."""
    B, C, C_a, H, W, K = shape
    d = synth.make_inputs(B, C, C_a, H, W, K, synth.BF16, seed=sum(shape), per_image_scale=True, channel_means=True)
    test_gpu_parity.compare_full(pkg, oracle, d, C_a, K, synth.BF16, synth.NHWC, what=f"{shape}")
    assert pkg.esc_convattn_last_path() == 4 and pkg.esc_convattn_last_tile_width() == 256 and pkg.esc_convattn_last_launches() == 2


@pytest.mark.parametrize("shape", [(64, 64, 32, 50, 130, 13, 8), (1, 64, 32, 700, 901, 7, 16)], ids=lambda s: "x".join(map(str, s)))
def test_forward_two_layer_estimator(pkg, oracle, shape):
    test_gpu_mlp.test_forward_mlp(pkg, oracle, shape, synth.BF16, synth.NHWC)
    assert pkg.esc_convattn_last_tile_width() == 256 and pkg.esc_convattn_last_launches() == 2


@pytest.mark.parametrize("case", [(64, 64, 32, 50, 130, 13, synth.BF16, synth.NHWC, True, "own"), (1, 48, 32, 700, 901, 13, synth.BF16, synth.NHWC, False, "x"),
                                  (20, 192, 48, 100, 150, 13, synth.BF16, synth.NHWC, True, "own")], ids=lambda c: "x".join(map(str, c[:6])))
def test_module(pkg, oracle, case):
    """Forward, 1x1 convolution and residual in one call: without the identity channels (C up to 128), and with them."""
    test_gpu_fuse.test_forward_fused(pkg, oracle, case)
    assert pkg.esc_convattn_last_tile_width() == 256 and pkg.esc_convattn_last_launches() == 3


def test_constant_of_the_backward_pass(pkg):
    """grad_x is this kernel on grad_out with rotated kernels and a constant per (image, channel): 1,200 small images against the
    same images in four calls, which take the kernel for smaller launches (each result one bf16 rounding: 2^-7 of its magnitude apart at most,
    and fp32 sums in another order)."""
    import torch

    B, C, C_a, H, W, K = 1200, 48, 32, 9, 40, 13
    d = synth.make_inputs(B, C, C_a, H, W, K, synth.BF16, seed=5, channel_means=True)
    x = util.to_device(d["x"], synth.BF16, synth.NHWC)
    wl, wd, bd = util.weights_to_device(d, synth.BF16)
    go = torch.randn(x.shape, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda").to(x.dtype)

    def run(x, go):
        gx = torch.empty_like(x)
        gl, gw, gb = (torch.zeros(t.shape, device="cuda") for t in (wl, wd, bd))
        ws = pkg.new_backward_workspace(x.shape[0], C_a, H, W, K)
        pkg.esc_convattn_backward(x, go, C_a, K, wl, wd, bd, gx, gl, gw, gb, pkg.ESC_NHWC, ws)
        torch.cuda.synchronize()
        assert pkg.esc_convattn_device_status(ws) == 0
        return gx, pkg.esc_convattn_last_tile_width()

    whole, width = run(x, go)
    assert width == 256
    for k in range(4):
        part, width = run(x[k * 300:k * 300 + 300].contiguous(), go[k * 300:k * 300 + 300].contiguous())
        assert width == 64
        a, b = whole[k * 300:k * 300 + 300].float(), part.float()
        assert torch.equal(a[..., C_a:], b[..., C_a:])
        assert bool(((a - b).abs() <= 2.0 ** -7 * torch.maximum(a.abs(), b.abs()) + 1e-4).all())


@pytest.mark.parametrize("K", [3, 9, 13])
def test_reach_of_a_non_finite_input(pkg, K):
    """Zero weights stand beside every tap, so accumulators outside the window become NaN; what is written does not."""
    import torch

    B, C, C_a, H, W = 700, 40, 32, 16, 40
    g = torch.Generator(device="cuda").manual_seed(K)

    def rand(*shape):
        t = torch.rand(shape, generator=g, device="cuda") + 0.25
        return t * (torch.randint(0, 2, shape, generator=g, device="cuda") * 2 - 1)

    x, w, dk = rand(B, H, W, C).bfloat16(), rand(C_a, K, K).bfloat16(), rand(B, C_a, 3, 3)
    ws = pkg.new_workspace(B, C_a, H, W, K)

    def run(x):
        out = torch.full_like(x, 7.0)
        pkg.esc_convattn_stencil(x, C_a, K, w, dk, out, pkg.ESC_NHWC, ws)
        torch.cuda.synchronize()
        assert pkg.esc_convattn_device_status(ws) == 0 and pkg.esc_convattn_last_tile_width() == 256
        return out

    want, P = run(x), K // 2
    for value, (b, c, y0, x0) in ((float("inf"), (B - 1, C_a - 1, 9, 20)), (float("nan"), (0, 1, 0, W - 1)), (float("-inf"), (7, 2, H - 1, 0))):
        xi = x.clone()
        xi[b, y0, x0, c] = value
        got = run(xi)
        reached = torch.zeros(got.shape, dtype=torch.bool, device="cuda")
        reached[b, max(0, y0 - P):y0 + P + 1, max(0, x0 - P):x0 + P + 1, c] = True
        assert bool((~torch.isfinite(got[reached])).all()), "an output does not see an input of its window"
        # outputs evaluated directly beside it: fp32 sums in another order, then one bf16 rounding
        a, b_ = got[~reached].float(), want[~reached].float()
        assert bool(torch.isfinite(a).all()) and bool(((a - b_).abs() <= 2.0 ** -7 * torch.maximum(a.abs(), b_.abs()) + 1e-4).all())


def by_definition(x, w, dk):
    """[B,H,W,C_a] in fp32 from bf16 x, w [C_a,K,K] and dk [B,C_a,3,3]: both sums tap by tap, so that IEEE arithmetic decides what a
    non-finite input does to the outputs of its window and nothing else."""
    import torch
    import torch.nn.functional as F

    H, W = x.shape[1:3]

    def taps(k, weight):
        P = k // 2
        pad = (0, 0, P, P, P, P)
        xp, inside = F.pad(x.float(), pad), F.pad(torch.ones(1, H, W, 1, dtype=torch.bool, device=x.device), pad)
        total = torch.zeros_like(x, dtype=torch.float32)
        for i in range(k):
            for j in range(k):
                total += torch.where(inside[:, i:i + H, j:j + W], xp[:, i:i + H, j:j + W] * weight(i, j), 0.0)
        return total

    return taps(w.shape[-1], lambda i, j: w[:, i, j].float()) + taps(3, lambda i, j: dk[:, None, None, :, i, j])


@pytest.mark.parametrize("K", [5, 13])
@pytest.mark.parametrize("what", ["nan", "inf", "one_channel", "every_16th", "inf_positive_taps", "nan_dk"])
def test_masses_of_non_finite_inputs(pkg, what, K):
    """Maps full of non-finite values: which outputs are NaN, the sign of the infinite ones, and the finite ones."""
    import torch

    B, C, C_a, H, W = 700, 40, 32, 16, 40
    g = torch.Generator(device="cuda").manual_seed(K)

    def rand(*shape):
        t = torch.rand(shape, generator=g, device="cuda") + 0.25
        return t * (torch.randint(0, 2, shape, generator=g, device="cuda") * 2 - 1)

    x, w, dk = rand(B, H, W, C).bfloat16(), rand(C_a, K, K).bfloat16(), rand(B, C_a, 3, 3)
    if what == "nan":
        x[..., :C_a] = float("nan")
    elif what == "inf":
        x[..., :C_a] = float("-inf")
    elif what == "inf_positive_taps":
        x[..., :C_a] = float("inf")
        w, dk = w.abs(), dk.abs()
    elif what == "one_channel":
        x[..., 5] = float("nan")
    elif what == "every_16th":
        x[:, ::16, ::16, :C_a] = float("inf")
    else:
        dk[3] = float("nan")
    ws = pkg.new_workspace(B, C_a, H, W, K)
    out = torch.full_like(x, 7.0)
    pkg.esc_convattn_stencil(x, C_a, K, w, dk, out, pkg.ESC_NHWC, ws)
    torch.cuda.synchronize()
    assert pkg.esc_convattn_device_status(ws) == 0 and pkg.esc_convattn_last_tile_width() == 256
    assert torch.equal(out[..., C_a:].view(torch.int16), x[..., C_a:].view(torch.int16))
    got, want = out[..., :C_a].float(), by_definition(x[..., :C_a], w, dk).bfloat16().float()
    assert torch.equal(torch.isnan(got), torch.isnan(want))
    assert torch.equal(torch.where(torch.isinf(got), got, 0.0), torch.where(torch.isinf(want), want, 0.0))
    a, b = got[torch.isfinite(got)], want[torch.isfinite(want)]
    # fp32 sums in another order, then one bf16 rounding
    assert a.numel() == 0 or bool(((a - b).abs() <= 2.0 ** -7 * torch.maximum(a.abs(), b.abs()) + 1e-4).all())


def test_time_does_not_hang_on_the_data(pkg):
    """One bad pixel, or a map of NaN, takes about as long as finite data.  (One 16-bit load after the other per output and tap, as it
    once was: 22 and 680 times as long.)"""
    import torch

    B, C, C_a, H, W, K = 1, 64, 32, 1080, 1920, 13
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn((B, H, W, C), generator=g, device="cuda").bfloat16()
    w = torch.randn((C_a, K, K), generator=g, device="cuda").bfloat16()
    dk = torch.randn((B, C_a, 3, 3), generator=g, device="cuda")
    out, ws = torch.empty_like(x), pkg.new_workspace(B, C_a, H, W, K)

    def time():
        best = float("inf")
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            pkg.esc_convattn_stencil(x, C_a, K, w, dk, out, pkg.ESC_NHWC, ws)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        assert pkg.esc_convattn_last_tile_width() == 256
        return best

    finite = time()
    x[0, 500, 900, 3] = float("inf")
    one = time()
    x[..., :C_a] = float("nan")
    everywhere = time()
    assert one < 6 * finite and everywhere < 2 * finite, (finite, one, everywhere)


def test_time_does_not_hang_on_the_width(pkg):
    """The identity channels are copied once whatever part of an image row a window takes: a pixel of 320-pixel rows costs about what
    one of 1,920-pixel rows does (1.06 times; 1.35 times when every part of a row was copied in whole chunks)."""
    import torch

    C, C_a, K = 64, 32, 13
    g = torch.Generator(device="cuda").manual_seed(2)
    w = torch.randn((C_a, K, K), generator=g, device="cuda").bfloat16()
    sides = []
    for B, H, W in ((16, 320, 320), (1, 1080, 1920)):
        x = torch.randn((B, H, W, C), generator=g, device="cuda").bfloat16()
        sides.append((x, torch.randn((B, C_a, 3, 3), generator=g, device="cuda"), torch.empty_like(x), pkg.new_workspace(B, C_a, H, W, K), B * H * W))
    best = [float("inf")] * 2
    for _ in range(8):
        for s, (x, dk, out, ws, pixels) in enumerate(sides):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            pkg.esc_convattn_stencil(x, C_a, K, w, dk, out, pkg.ESC_NHWC, ws)
            a.record()
            for _ in range(4):
                pkg.esc_convattn_stencil(x, C_a, K, w, dk, out, pkg.ESC_NHWC, ws)
            b.record()
            torch.cuda.synchronize()
            assert pkg.esc_convattn_last_tile_width() == 256
            best[s] = min(best[s], a.elapsed_time(b) / pixels)
    assert best[0] < 1.25 * best[1], best


@pytest.mark.parametrize("shape", [(64, 40, 32, 64, 160), (128, 96, 96, 40, 40)], ids=lambda s: "x".join(map(str, s)))
def test_pooling_grid_is_the_same_for_every_kernel_size(pkg, shape):
    """The pooling kernel in front takes the grid of a batch whatever K is: the workspace (dk, partial sums) comes out bit for bit the
    same for K = 13, 9 and 3 on the same map."""
    import torch

    B, C, C_a, H, W = shape
    d = synth.make_inputs(B, C, C_a, H, W, 13, synth.BF16, seed=11, channel_means=True)
    x = util.to_device(d["x"], synth.BF16, synth.NHWC)
    wl, wd, bd = util.weights_to_device(d, synth.BF16)
    left = []
    for K in (13, 9, 3):
        off = (13 - K) // 2
        ws = pkg.new_workspace(B, C_a, H, W, K).zero_()
        pkg.esc_convattn_forward_ex(x, C_a, K, wl[:, off:off + K, off:off + K].contiguous(), wd, bd, torch.empty_like(x), pkg.ESC_NHWC, ws)
        torch.cuda.synchronize()
        assert pkg.esc_convattn_device_status(ws) == 0 and pkg.esc_convattn_last_tile_width() == 256
        left.append(ws)
    assert bool((left[0] != 0).any()) and torch.equal(left[0], left[1]) and torch.equal(left[0], left[2])

"""GPU parity of the FP32 tap-gradient kernels (the chain rule of the ESC paper's Eq. 4) where the way they share the 13 kernel rows
changes: one block per tile and channel with 512 or 128 threads (NCHW), up to four blocks per tile (NHWC), ragged tiles, several
tiles per image, kernel sizes below 13.

Bars: fp32 sums of B*H*W products in any order, 1e-5 of the sum of magnitudes."""
import pytest

from paper_2503_06671_b200 import synth

pytestmark = pytest.mark.gpu

CASES = [
    # B, C, C_a, H, W, K
    (1, 8, 8, 5, 3, 13), (2, 16, 16, 64, 64, 13), (3, 24, 16, 65, 97, 9), (18, 16, 16, 64, 64, 13),   # 1, 32, 192 and 288 tiles of a channel
    (19, 16, 16, 63, 33, 13), (10, 40, 40, 41, 41, 13), (9, 16, 16, 33, 70, 13),                       # 304, 400, 288
]


@pytest.mark.parametrize("layout", [synth.NCHW, synth.NHWC], ids=["nchw", "nhwc"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_tap_gradients(case, layout):
    import torch
    import torch.nn.functional as F

    import paper_2503_06671_b200 as pkg

    B, C, C_a, H, W, K = case
    g = torch.Generator(device="cuda").manual_seed(sum(case))
    x, go = (torch.randn((B, C, H, W), generator=g, device="cuda") + 0.1 for _ in range(2))
    wl = torch.randn((C_a, K, K), generator=g, device="cuda") / K
    wd, bd = torch.randn((9 * C_a, C_a), generator=g, device="cuda") / C_a, torch.randn((9 * C_a,), generator=g, device="cuda")
    chl = layout == synth.NHWC
    xl, gl = (t.permute(0, 2, 3, 1).contiguous() if chl else t for t in (x, go))
    gx, g_lk, g_wd, g_bd = torch.empty_like(xl), torch.zeros_like(wl), torch.zeros_like(wd), torch.zeros_like(bd)
    ws = pkg.new_backward_workspace(B, C_a, H, W, K)
    for _ in range(2):
        pkg.esc_convattn_backward(xl, gl, C_a, K, wl, wd, bd, gx, g_lk, g_wd, g_bd, pkg.ESC_NHWC if chl else pkg.ESC_NCHW, ws)
    torch.cuda.synchronize()

    def taps(a, b):                                       # [B][C_a][13][13]: sum over the map of b times a, shifted
        a = F.pad(a[:, :C_a].double(), (6, 6, 6, 6))
        return torch.stack([(a[:, :, i:i + H, j:j + W] * b[:, :C_a].double()).sum((2, 3)) for i in range(13) for j in range(13)], 2).view(B, C_a, 13, 13)

    t, m = taps(x, go), taps(x.abs(), go.abs())
    lo, hi = (13 - K) // 2, 13 - (13 - K) // 2
    assert bool(((g_lk - t.sum(0)[:, lo:hi, lo:hi]).abs() <= 1e-5 * m.sum(0)[:, lo:hi, lo:hi]).all())
    gdk, mdk = t[:, :, 5:8, 5:8].reshape(B, -1), m[:, :, 5:8, 5:8].reshape(B, -1)
    assert bool(((g_bd - gdk.sum(0)).abs() <= 1e-5 * mdk.sum(0)).all())
    mean, amean = x[:, :C_a].double().mean((2, 3)), x[:, :C_a].double().abs().mean((2, 3))
    assert bool(((g_wd - gdk.T @ mean).abs() <= 2e-5 * (mdk.T @ amean)).all())


@pytest.mark.parametrize("layout", [synth.NCHW, synth.NHWC], ids=["nchw", "nhwc"])
@pytest.mark.parametrize("dtype", [synth.F32, synth.BF16], ids=["fp32", "bf16"])
def test_without_the_large_kernels_gradient(dtype, layout):
    """Without g_lk only the middle kernel rows are formed: the other gradients keep their bits."""
    import torch

    import paper_2503_06671_b200 as pkg

    B, C, C_a, H, W, K = 3, 32, 16, 37, 136, 13
    g = torch.Generator(device="cuda").manual_seed(7)
    dt = torch.bfloat16 if dtype == synth.BF16 else torch.float32
    x, go = (torch.randn((B, C, H, W) if layout == synth.NCHW else (B, H, W, C), generator=g, device="cuda").to(dt) for _ in range(2))
    wl, wd, bd = (torch.randn(s, generator=g, device="cuda").to(dt) / 13 for s in ((C_a, K, K), (9 * C_a, C_a), (9 * C_a,)))
    res = []
    for lk in (torch.zeros((C_a, K, K), device="cuda"), None):
        gx, g_wd, g_bd = torch.empty_like(x), torch.zeros(wd.shape, device="cuda"), torch.zeros(bd.shape, device="cuda")
        ws = pkg.new_backward_workspace(B, C_a, H, W, K)
        pkg.esc_convattn_backward(x, go, C_a, K, wl, wd, bd, gx, lk, g_wd, g_bd, pkg.ESC_NHWC if layout == synth.NHWC else pkg.ESC_NCHW, ws)
        torch.cuda.synchronize()
        res.append((gx, g_wd, g_bd))
    assert all(torch.equal(a, b) for a, b in zip(*res))

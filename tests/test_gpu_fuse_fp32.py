"""GPU parity of the closing 1x1 convolution on the FP32 pipe, forward (inside the module) and backward, against the CPU oracle:
pixel counts around its tiles of 128 and passes of 64, images whose planes are not whole 16-byte pieces, every width it is
compiled for, identity channels taken from x at a split that is not a whole 16-byte piece.

Bars as in test_gpu_fuse.py and test_gpu_fuse_backward.py: 1e-5 of the sum of magnitudes for fp32 sums, beside the rounding
of a bf16 result (2^-8) and of the bf16 map between the two kernels."""
import numpy as np
import pytest

from paper_2503_06671_b200 import synth
from tests import util

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import paper_2503_06671_b200 as p

    p.lib()
    return p


CASES = [
    # B, C, C_a, H, W, dtype
    (1, 16, 8, 1, 1, synth.F32),         # one pixel
    (2, 32, 16, 9, 7, synth.F32),        # 63 pixels an image: not whole 16-byte pieces, less than a tile
    (2, 48, 6, 8, 16, synth.F32),        # exactly one tile an image; attention channels end inside a 16-byte piece
    (1, 64, 16, 3, 43, synth.F32),       # 129 pixels
    (3, 64, 16, 33, 52, synth.F32),
    (2, 64, 16, 13, 21, synth.BF16),     # NCHW: 273 pixels an image, which the tensor-core kernels do not take
    (1, 16, 16, 17, 19, synth.BF16),
]


@pytest.mark.parametrize("layout", [synth.NCHW, synth.NHWC])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_fuse_fp32_pipe(pkg, oracle, case, layout):
    import torch

    B, C, C_a, H, W, dtype = case
    K = 13
    seed = sum(case[:5])
    d = synth.make_inputs(B, C, C_a, H, W, K, dtype, seed=seed, per_image_scale=True, channel_means=True)
    f = synth.make_fuse(C, dtype, seed=seed)
    rng = np.random.default_rng(seed)
    res, go = (synth.round_to(rng.normal(size=d["x"].shape).astype(np.float32), dtype) for _ in range(2))
    tdt = util.torch_dtype(dtype)
    x, rd, god = (util.to_device(a, dtype, layout) for a in (d["x"], res, go))
    wl, wd, bd = util.weights_to_device(d, dtype)
    wf, bf = (torch.from_numpy(f[k]).to("cuda", tdt) for k in ("w_fuse", "b_fuse"))
    code = util.layout_code(layout)
    n = x.numel()
    buf = torch.full((n + 2048,), 7.0, dtype=x.dtype, device="cuda")
    out = buf[1024:1024 + n].view(x.shape)
    ws = pkg.new_workspace(B, C_a, H, W, K)
    pkg.esc_convattn_forward_fused(x, C_a, K, wl, wd, bd, wf, bf, rd, out, code, ws)
    torch.cuda.synchronize()
    assert bool((buf[:1024] == 7.0).all()) and bool((buf[1024 + n:] == 7.0).all()), "write outside out"
    ref, mag, cat = oracle.forward_fused(d["x"], C_a, d["w_large"], d["w_dyn"], d["b_dyn"], f["w_fuse"], f["b_fuse"], res,
                                         want_mag=True, want_cat=True)
    err = np.abs(util.to_host_nchw(out, layout).astype(np.float64) - ref)
    bar = 1e-5 * mag + 1e-30
    if dtype == synth.BF16:
        carried = np.einsum("nc,bchw->bnhw", np.abs(f["w_fuse"][:, :C_a]).astype(np.float64), np.abs(cat[:, :C_a]))
        bar = bar + 2.0 ** -8 * np.abs(ref) * 1.001 + 2.0 ** -8 * carried
    assert (err <= bar).all(), f"forward, worst {(err / bar).max():.2f} bars"

    g_cat = torch.full_like(x, 7.0)
    g_w = torch.full((C, C), float("nan"), device="cuda")
    g_b = torch.full((C,), float("nan"), device="cuda")
    pkg.esc_conv_fuse_backward(x, god, wf, g_cat, g_w, g_b, code)
    torch.cuda.synchronize()
    go64, x64, w64 = (a.astype(np.float64) for a in (go, d["x"], f["w_fuse"]))
    for got, a, b, spec in ((g_w, go64, x64, "bnhw,bchw->nc"), (g_b, go64, np.ones_like(x64), "bnhw,bnhw->n")):
        want, scale = np.einsum(spec, a, b), np.einsum(spec, np.abs(a), np.abs(b))
        assert (np.abs(got.cpu().numpy() - want) <= 1e-5 * scale + 1e-30).all()
    want, scale = np.einsum("nc,bnhw->bchw", w64, go64), np.einsum("nc,bnhw->bchw", np.abs(w64), np.abs(go64))
    err = np.abs(util.to_host_nchw(g_cat, layout) - want)
    bar = 1e-5 * scale + 1e-30 + (2.0 ** -8 * np.abs(want) * 1.001 if dtype == synth.BF16 else 0.0)
    assert (err <= bar).all(), f"g_cat, worst {(err / bar).max():.2f} bars"

"""GPU parity of the estimator's part of the backward pass (ESC paper, Eq. 4 line 2, differentiated) where its kernels change
their way: tap gradients added up on the way (up to 16 tiles an image) or by a kernel of their own, more images than warps of a
block, widths of one and of the largest hidden layer, channel counts that do not fill a warp and that do not fit shared memory.

Bars as in test_gpu_backward.py and test_gpu_backward_mlp.py: 1e-5 (one layer) and 2e-5 (two) of the sums' scale."""
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
    # B, C, C_a, H, W, hidden, dtype, layout
    (1, 16, 16, 256, 24, 0, synth.BF16, synth.NHWC),      # 16 tiles of 64x16: added up on the way
    (1, 16, 16, 272, 24, 0, synth.BF16, synth.NHWC),      # 17: by sum_tiles
    (1, 16, 16, 272, 24, 8, synth.BF16, synth.NCHW),
    (9, 16, 16, 20, 24, 1, synth.BF16, synth.NHWC),       # more images than warps; one hidden unit
    (33, 24, 5, 12, 10, 0, synth.F32, synth.NCHW),        # 45 estimator outputs
    (17, 16, 3, 9, 10, 128, synth.F32, synth.NHWC),       # the widest hidden layer
    (2, 1100, 1100, 5, 6, 0, synth.F32, synth.NCHW),      # more channels than shared memory has room for
    # few images, whose weight gradients come from the same kernel: the most of them, with one and two layers, the most channels, and
    # the next count, whose do not
    (8, 16, 16, 200, 40, 0, synth.BF16, synth.NHWC),      # 13 tiles an image, added up on the way
    (2, 16, 16, 280, 24, 8, synth.BF16, synth.NCHW),      # 18, by sum_tiles
    (4, 256, 256, 6, 7, 0, synth.F32, synth.NCHW),
    (1, 24, 5, 12, 10, 16, synth.F32, synth.NHWC),
    (1, 24, 5, 12, 10, 17, synth.F32, synth.NHWC),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_estimator_gradients(pkg, oracle, case):
    import torch

    B, C, C_a, H, W, h, dtype, layout = case
    K = 13
    seed = sum(case[:6])
    d = synth.make_inputs(B, C, C_a, H, W, K, dtype, seed=seed, per_image_scale=True, channel_means=True)
    go = synth.round_to(np.random.default_rng(seed).standard_normal(size=d["x"].shape).astype(np.float32), dtype)
    tdt, code = util.torch_dtype(dtype), util.layout_code(layout)
    x, god = util.to_device(d["x"], dtype, layout), util.to_device(go, dtype, layout)
    gx = torch.empty_like(x)
    ws = pkg.new_backward_workspace(B, C_a, H, W, K)
    ax, ago = np.abs(d["x"]), np.abs(go)

    def nan(*shape):
        return torch.full(shape, float("nan"), device="cuda")

    if h == 0:
        wl, wd, bd = util.weights_to_device(d, dtype)
        got = [nan(C_a, K, K), nan(9 * C_a, C_a), nan(9 * C_a)]
        pkg.esc_convattn_backward(x, god, C_a, K, wl, wd, bd, gx, *got, code, ws)
        ref = oracle.backward(d["x"], go, C_a, d["w_large"], d["w_dyn"], d["b_dyn"])
        scale = oracle.backward(ax, ago, C_a, d["w_large"], d["w_dyn"], d["b_dyn"])[1:]
        tol, const = 1e-5, 1e-5 * np.abs(d["w_dyn"]).astype(np.float64).T @ scale[2] / (H * W)
        dk = oracle.dynkernel(oracle.gap(d["x"], C_a), d["w_dyn"], d["b_dyn"])
    else:
        keys = ("w_down", "b_down", "w_up", "b_up")
        m = synth.make_estimator_mlp(C_a, h, dtype, seed=seed)
        wl = torch.from_numpy(d["w_large"]).to("cuda", tdt)
        got = [nan(C_a, K, K), nan(h, C_a), nan(h), nan(9 * C_a, h), nan(9 * C_a)]
        pkg.esc_convattn_backward_mlp(x, god, C_a, K, wl, *(torch.from_numpy(m[k]).to("cuda", tdt) for k in keys), gx, *got, code, ws)
        ref = oracle.backward_mlp(d["x"], go, C_a, d["w_large"], *(m[k] for k in keys))
        mean = np.abs(oracle.gap(ax, C_a))
        _, alk, _, ab = oracle.backward(ax, ago, C_a, d["w_large"], np.zeros((9 * C_a, C_a)), np.zeros(9 * C_a))
        act = np.abs(mean @ np.abs(m["w_down"]).T + np.abs(m["b_down"])).max(axis=0)          # |phi(t)| <= |t|
        s_bd = 1.13 * (ab @ np.abs(m["w_up"]))                                                # |phi'| <= 1.13
        scale = [alk, np.outer(s_bd, mean.max(axis=0)), s_bd, np.outer(ab, act), ab]
        tol, const = 2e-5, 2e-5 * (s_bd @ np.abs(m["w_down"])) / (H * W)
        dk = oracle.dynkernel_mlp(oracle.gap(d["x"], C_a), *(m[k] for k in keys))
    torch.cuda.synchronize()
    assert pkg.esc_convattn_device_status(ws) == 0
    for g, r, s in zip(got, ref[1:], scale):
        err = np.abs(g.cpu().numpy().astype(np.float64) - r)
        assert (err <= tol * s + 1e-30).all(), f"worst {(err / np.maximum(s, 1e-30)).max():.3e} of its scale"
    mag = oracle.stencil(ago, C_a, np.abs(d["w_large"][:, ::-1, ::-1]).copy(), np.abs(dk[:, :, ::-1, ::-1]).copy())[:, :C_a]
    out = util.to_host_nchw(gx, layout)
    err = np.abs(out[:, :C_a] - ref[0][:, :C_a])
    bar = 1e-5 * mag + const[None, :, None, None] + 1e-30
    if dtype == synth.BF16:
        bar = bar + 2.0 ** -8 * np.abs(ref[0][:, :C_a]) * 1.001
    assert (err <= bar).all()

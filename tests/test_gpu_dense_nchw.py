"""GPU parity of the dense large kernel (ESC paper, Section 3.2) on bf16 NCHW tensors behind the packing pass: maps of at least
4,096 pixels of any width, forward, the stage alone, and every gradient.

Bars as in test_gpu_dense.py and test_gpu_backward_dense.py: one rounding of a result (2^-8), 5e-5 of the sum of magnitudes on the
tensor cores, 1e-5 for the weight gradients."""
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
    # B, C, H, W, K, path
    (1, 24, 64, 64, 13, 5),       # the fewest pixels that are packed
    (1, 24, 63, 65, 13, 1),       # one less: the FP32-pipe kernel
    (2, 16, 37, 59, 13, 5),       # odd sizes, images start at odd elements, nothing to copy through
    (3, 20, 45, 33, 9, 5),        # identity planes that are not whole 16-byte pieces
    (1, 64, 20, 300, 3, 5),       # three strips
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_dense_nchw(pkg, oracle, case):
    import torch

    B, C, H, W, K, path = case
    C_a = 16
    seed = sum(case)
    d = synth.make_inputs(B, C, C_a, H, W, K, synth.BF16, seed=seed, per_image_scale=True, channel_means=True)
    wdn = synth.make_dense_kernel(C_a, K, synth.BF16, seed=seed)
    go = synth.round_to(np.random.default_rng(seed).standard_normal(size=d["x"].shape).astype(np.float32), synth.BF16)
    x, god = util.to_device(d["x"], synth.BF16, synth.NCHW), util.to_device(go, synth.BF16, synth.NCHW)
    _, wd, bd = util.weights_to_device(d, synth.BF16)
    wdd = torch.from_numpy(wdn).to("cuda", torch.bfloat16)
    n = x.numel()
    buf = torch.full((n + 2048,), 7.0, dtype=x.dtype, device="cuda")
    out = buf[1024:1024 + n].view(x.shape)

    def check(got, ref, mag, what):
        got = util.to_host_nchw(got, synth.NCHW)
        err = np.abs(got[:, :C_a] - ref[:, :C_a])
        bar = 2.0 ** -8 * np.abs(ref[:, :C_a]) * 1.001 + 5e-5 * mag[:, :C_a] + 1e-30
        assert (err <= bar).all(), f"{what}: worst {(err / bar).max():.2f} bars"
        assert np.array_equal(got[:, C_a:], ref[:, C_a:]), what
        assert bool((buf[:1024] == 7.0).all()) and bool((buf[1024 + n:] == 7.0).all()), "write outside out"

    ws = pkg.new_workspace(B, C_a, H, W, K)
    for _ in range(2):
        pkg.esc_convattn_forward_dense(x, C_a, K, wdd, wd, bd, out, pkg.ESC_NCHW, ws)
    torch.cuda.synchronize()
    assert pkg.esc_convattn_device_status(ws) == 0 and pkg.esc_convattn_last_path() == path
    check(out, *oracle.forward_dense(d["x"], C_a, wdn, d["w_dyn"], d["b_dyn"], want_mag=True), "forward")
    dk = np.random.default_rng(7).uniform(-0.5, 0.5, size=(B, C_a, 3, 3)).astype(np.float32)
    out.fill_(7.0)
    pkg.esc_convattn_stencil_dense(x, C_a, K, wdd, torch.from_numpy(dk).cuda(), out, pkg.ESC_NCHW, ws)
    torch.cuda.synchronize()
    check(out, *oracle.stencil_dense(d["x"], C_a, wdn, dk, want_mag=True), "stage alone")

    wsb = pkg.new_backward_dense_workspace(B, C_a, H, W, K)
    g = [torch.full(s, float("nan"), device="cuda") for s in ((C_a, C_a, K, K), (9 * C_a, C_a), (9 * C_a,))]
    out.fill_(7.0)
    for _ in range(2):
        pkg.esc_convattn_backward_dense(x, god, C_a, K, wdd, wd, bd, out, *g, pkg.ESC_NCHW, wsb)
    torch.cuda.synchronize()
    assert pkg.esc_convattn_device_status(wsb) == 0
    ref = oracle.backward_dense(d["x"], go, C_a, wdn, d["w_dyn"], d["b_dyn"])
    mag = oracle.backward_dense(np.abs(d["x"]), np.abs(go), C_a, np.abs(wdn), np.abs(d["w_dyn"]), np.abs(d["b_dyn"]))
    if path == 5:
        check(out, ref[0], mag[0], "grad x")
    for name, got, r, s in zip(("w_dense", "w_dyn", "b_dyn"), g, ref[1:], mag[1:]):
        err = np.abs(got.cpu().numpy().astype(np.float64) - r)
        assert (err <= 1e-5 * s + 1e-30).all(), f"grad {name}: worst {(err / np.maximum(s, 1e-30)).max():.3e} of its scale"


def test_workspace_without_room_for_packed_maps(pkg):
    """The packed maps are the last part of a workspace (32 bytes per pixel forward, 64 backward) and may be missing: the same calls
    then run on the kernels that need none, forward, stage alone and gradients.  One byte less is refused."""
    import torch

    B, C, C_a, H, W, K = 2, 24, 16, 50, 60, 13
    d = synth.make_inputs(B, C, C_a, H, W, K, synth.BF16, seed=5, channel_means=True)
    x, god = (util.to_device(a, synth.BF16, synth.NCHW) for a in (d["x"], synth.round_to(d["x"][::-1].copy(), synth.BF16)))
    _, wd, bd = util.weights_to_device(d, synth.BF16)
    wdd = torch.from_numpy(synth.make_dense_kernel(C_a, K, synth.BF16, seed=5)).to("cuda", torch.bfloat16)
    dk = torch.rand(B, C_a, 3, 3, device="cuda") - 0.5
    part = -(-B * H * W * 32 // 256) * 256
    res = {}
    for room in (True, False):
        ws, wsb = pkg.new_workspace(B, C_a, H, W, K), pkg.new_backward_dense_workspace(B, C_a, H, W, K)
        if not room:
            ws, wsb = ws[:ws.numel() - part], wsb[:wsb.numel() - 2 * part]
        o = [torch.full_like(x, 7.0) for _ in range(3)]
        g = [torch.full(s, float("nan"), device="cuda") for s in ((C_a, C_a, K, K), (9 * C_a, C_a), (9 * C_a,))]
        paths = []
        pkg.esc_convattn_forward_dense(x, C_a, K, wdd, wd, bd, o[0], pkg.ESC_NCHW, ws)
        paths.append(pkg.esc_convattn_last_path())
        pkg.esc_convattn_stencil_dense(x, C_a, K, wdd, dk, o[1], pkg.ESC_NCHW, ws)
        paths.append(pkg.esc_convattn_last_path())
        pkg.esc_convattn_backward_dense(x, god, C_a, K, wdd, wd, bd, o[2], *g, pkg.ESC_NCHW, wsb)
        paths.append(pkg.esc_convattn_last_path())
        torch.cuda.synchronize()
        assert pkg.esc_convattn_device_status(ws) == 0 and pkg.esc_convattn_device_status(wsb) == 0
        assert paths == [5 if room else 1] * 3
        res[room] = o + g
        if not room:
            with pytest.raises(pkg.EscError):
                pkg.esc_convattn_forward_dense(x, C_a, K, wdd, wd, bd, o[0], pkg.ESC_NCHW, ws[:-1])
            with pytest.raises(pkg.EscError):
                pkg.esc_convattn_backward_dense(x, god, C_a, K, wdd, wd, bd, o[2], *g, pkg.ESC_NCHW, wsb[:-1])
    # maps: fp32 sums in another order (5e-5 of magnitudes of about 10), one rounding each: at most one bf16 step apart; weight gradients:
    # 1e-5 of the scale on either side
    for a, b in zip(res[True][:3], res[False][:3]):
        diff, size = (a.float() - b.float()).abs(), b.float().abs()
        assert bool((diff <= 2.0 ** -7 * size + 1e-3).all()) and torch.equal(a[:, C_a:], b[:, C_a:])
    for a, b in zip(res[True][3:], res[False][3:]):
        assert float((a - b).abs().max()) <= 2e-5 * float(b.abs().max())

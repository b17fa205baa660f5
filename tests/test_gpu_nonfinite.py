"""A non-finite input reaches the outputs whose window holds it and no others, for every kernel size of the kernels that promise it: the
register-tiled FP32 stencil (either layout, one and four channels a block, with the point-wise mix), the dense form on the FP32 pipe and
on tcgen05 (NHWC, and NCHW behind the packing pass).  Stage 2 alone, so that the pooled means do not spread it.  (The banded Toeplitz
kernels sum 16 neighbours in one instruction; their reach is stated in the header.)"""
import pytest

from paper_2503_06671_b200 import synth
from tests import util

pytestmark = pytest.mark.gpu

CASES = [
    # form, dtype, layout, B, C, C_a, H, W, path
    ("depthwise", synth.F32, synth.NCHW, 1, 7, 5, 40, 50, 1),
    ("depthwise", synth.F32, synth.NCHW, 2, 20, 16, 150, 300, 1),
    ("depthwise", synth.F32, synth.NHWC, 2, 20, 16, 45, 70, 1),
    ("depthwise", synth.BF16, synth.NCHW, 1, 24, 16, 45, 70, 1),       # too few units for the tensor-core kernel
    ("decomposed", synth.F32, synth.NHWC, 1, 20, 8, 45, 70, 1),
    ("decomposed", synth.F32, synth.NCHW, 1, 20, 8, 45, 70, 1),
    ("dense", synth.F32, synth.NCHW, 1, 20, 16, 45, 70, 1),
    ("dense", synth.F32, synth.NHWC, 2, 20, 16, 150, 300, 1),
    ("dense", synth.BF16, synth.NHWC, 2, 24, 16, 75, 150, 5),          # K <= 13
    ("dense", synth.BF16, synth.NCHW, 2, 20, 16, 75, 150, 5),          # K <= 13
]


@pytest.mark.parametrize("K", [3, 5, 7, 9, 11, 13, 15, 17])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
def test_reach_of_a_non_finite_input(case, K):
    import torch

    import paper_2503_06671_b200 as pkg

    form, dtype, layout, B, C, C_a, H, W, path = case
    tdt, lay = util.torch_dtype(dtype), util.layout_code(layout)
    g = torch.Generator(device="cuda").manual_seed(K)

    def rand(*shape):
        t = torch.rand(shape, generator=g, device="cuda") + 0.25       # no zero weight
        return (t * (torch.randint(0, 2, shape, generator=g, device="cuda") * 2 - 1)).to(tdt)

    x = rand(B, C, H, W)
    w = rand(C_a, C_a, K, K) if form == "dense" else rand(C_a, K, K)
    w_point = rand(C_a, C_a)
    dk = rand(B, C_a, 3, 3).float()
    ws = pkg.new_workspace(B, C_a, H, W, K)

    def run(x):
        xm = x.permute(0, 2, 3, 1).contiguous() if layout == synth.NHWC else x
        out = torch.full_like(xm, 7.0)
        if form == "dense":
            pkg.esc_convattn_stencil_dense(xm, C_a, K, w, dk, out, lay, ws)
        elif form == "decomposed":
            pkg.esc_convattn_stencil_pw(xm, C_a, K, w, w_point, dk, out, lay, ws)
        else:
            pkg.esc_convattn_stencil(xm, C_a, K, w, dk, out, lay, ws)
        torch.cuda.synchronize()
        assert pkg.esc_convattn_device_status(ws) == 0
        assert pkg.esc_convattn_last_path() == (path if K <= 13 else 1)
        return out.permute(0, 3, 1, 2) if layout == synth.NHWC else out

    want, P = run(x), (K - 1) // 2
    for value, (b, c, y0, x0) in ((float("inf"), (B - 1, C_a - 1, H // 2 + 1, W // 2 + 3)), (float("nan"), (0, 1, 0, W - 1)),
                                  (float("-inf"), (0, 2, H - 1, 31))):
        xi = x.clone()
        xi[b, c, y0, x0] = value
        got = run(xi)
        reached = torch.zeros(got.shape, dtype=torch.bool, device="cuda")
        channels = slice(c, c + 1) if form == "depthwise" else slice(0, C_a)
        reached[b, channels, max(0, y0 - P):y0 + P + 1, max(0, x0 - P):x0 + P + 1] = True
        assert bool((~torch.isfinite(got[reached])).all()), "an output does not see an input of its window"
        assert torch.equal(got[~reached], want[~reached]), "an output sees an input outside its window"

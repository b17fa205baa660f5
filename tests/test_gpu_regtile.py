"""GPU parity of the register-tiled stencils (ESC paper, Eq. 4 lines 3-4; Eq. 5 with the point-wise mix): each kernel size that is
padded to the next one built, one and four channels per block, both geometries, tiles that end inside the image, element types.

Bars: fp32 sums of K*K (with the mix C_a*K*K) terms in any order, 1e-5 of the sum of magnitudes; bf16 results also one rounding."""
import numpy as np
import pytest

from paper_2503_06671_b200 import synth

pytestmark = pytest.mark.gpu

CASES = [
    # B, C, C_a, H, W, K, mix
    *[(1, 8, 4, 33, 65, k, False) for k in (3, 5, 7, 9, 11, 13, 15, 17)],
    (2, 9, 5, 31, 32, 17, False), (1, 8, 8, 1, 1, 9, False),        # an odd number of channels; a single pixel
    (1, 12, 12, 32, 64, 13, True), (1, 7, 6, 35, 67, 13, True), (3, 20, 16, 34, 66, 9, True), (1, 8, 4, 40, 70, 17, True),
    (2, 40, 36, 161, 321, 13, False), (2, 36, 36, 161, 321, 9, True),   # larger launches: several blocks on every SM
]


@pytest.mark.parametrize("layout", [synth.NCHW, synth.NHWC], ids=["nchw", "nhwc"])
@pytest.mark.parametrize("dtype", [synth.F32, synth.BF16], ids=["fp32", "bf16"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_register_tiles(case, dtype, layout):
    import torch
    import torch.nn.functional as F

    import paper_2503_06671_b200 as pkg

    B, C, C_a, H, W, K, mix = case
    g = torch.Generator(device="cuda").manual_seed(sum(case))
    dt = torch.bfloat16 if dtype == synth.BF16 else torch.float32
    x = torch.randn((B, C, H, W), generator=g, device="cuda").to(dt)
    wl = (torch.randn((C_a, K, K), generator=g, device="cuda") / K).to(dt)
    wp = (torch.randn((C_a, C_a), generator=g, device="cuda") / C_a ** 0.5).to(dt) if mix else None
    dk = torch.randn((B, C_a, 9), generator=g, device="cuda")

    def stage(x, wl, wp, dk):
        m = x[:, :C_a]
        if mix:
            m = F.conv2d(m, wp[:, :, None, None])
        y = F.conv2d(m, wl[:, None], padding=K // 2, groups=C_a)
        return y + F.conv2d(m.reshape(1, B * C_a, H, W), dk.reshape(B * C_a, 1, 3, 3), padding=1, groups=B * C_a).reshape(B, C_a, H, W)

    args = [None if t is None else t.double() for t in (x, wl, wp, dk)]
    want, mag = stage(*args), stage(*[None if t is None else t.abs() for t in args])
    chl = layout == synth.NHWC
    xl = x.permute(0, 2, 3, 1).contiguous() if chl else x
    out = torch.full_like(xl, 7.0)
    code = pkg.ESC_NHWC if chl else pkg.ESC_NCHW
    if mix:
        pkg.esc_convattn_stencil_pw(xl, C_a, K, wl, wp, dk, out, code)
    else:
        pkg.esc_convattn_stencil(xl, C_a, K, wl, dk, out, code)
    torch.cuda.synchronize()
    path = pkg.esc_convattn_last_path()
    assert path == 1 or dtype == synth.BF16
    got = out.permute(0, 3, 1, 2) if chl else out
    assert torch.equal(got[:, C_a:], x[:, C_a:])
    bar = 1e-5 * mag + ((2.0 ** -8 * want.abs() + (2.0 ** -8 * mag if path != 1 and mix else 0)) if dtype == synth.BF16 else 0)
    assert bool(((got[:, :C_a].double() - want).abs() <= bar).all())

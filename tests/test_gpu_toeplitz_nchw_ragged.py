"""GPU parity of the NCHW tensor-core kernel on widths that are not a multiple of 8 (ESC paper, Eq. 4 lines 3-4; Eq. 5 with the
point-wise mix): every residue of the width modulo 8, one and several units per CTA with buffers re-used, stage 1 inside the
launch and before it, two channel groups, the last row and pixel of the tensor, guard bands around the output.

Bars: one rounding of the result (2^-8) and fp32 noise (1e-5 of the sum of magnitudes); with the mix also what the mixed map's
high and low half leave out (2^-16 of the sum of magnitudes): far less than the 2^-8 of a mixed map rounded to bf16."""
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
    # B, C, C_a, H, W, K, decomposed
    *[(1, 24, 16, 130, 320 + r, 13, False) for r in range(1, 8)],   # every residue; 54 units
    (60, 16, 16, 9, 5, 13, False),         # rows shorter than one piece, nothing to copy through
    (25, 24, 16, 7, 65, 13, True),         # a second tile of one column
    (1, 48, 16, 240, 427, 13, True),
    (1, 32, 16, 250, 163, 9, True),        # K = 9 padded to 13; 48 units, the fewest
    (3, 40, 32, 200, 301, 13, False),      # 390 units: two channel groups, two or three units per CTA
    (12, 24, 16, 199, 331, 13, True),      # 936 units: six or seven per CTA, images change inside a CTA's walk
    (2, 64, 16, 201, 511, 13, False),      # 208 units: one or two per CTA, one launch
]


@pytest.mark.parametrize("one_launch", [True, False])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_ragged_widths(pkg, oracle, case, one_launch):
    import torch

    B, C, C_a, H, W, K, mix = case
    seed = sum(case[:6])
    d = synth.make_inputs(B, C, C_a, H, W, K, synth.BF16, seed=seed, per_image_scale=True, channel_means=True)
    x = util.to_device(d["x"], synth.BF16, synth.NCHW)
    wl, wd, bd = util.weights_to_device(d, synth.BF16)
    n = x.numel()
    buf = torch.full((n + 2048,), 7.0, dtype=x.dtype, device="cuda")
    out = buf[1024:1024 + n].view(x.shape)
    ws = pkg.new_workspace(B, C_a, H, W, K)
    wp = synth.round_to(np.random.default_rng(seed).uniform(-0.25, 0.25, (C_a, C_a)).astype(np.float32), synth.BF16) if mix else None
    pkg.esc_convattn_set_fused_stage1(one_launch)
    try:
        for _ in range(2):                                  # twice: barriers and buffers start clean each launch
            if mix:
                pkg.esc_convattn_forward_pw(x, C_a, K, wl, torch.from_numpy(wp).to("cuda", torch.bfloat16), wd, bd, out, pkg.ESC_NCHW, ws)
            else:
                pkg.esc_convattn_forward_ex(x, C_a, K, wl, wd, bd, out, pkg.ESC_NCHW, ws)
        torch.cuda.synchronize()
    finally:
        pkg.esc_convattn_set_fused_stage1(True)
    assert pkg.esc_convattn_device_status(ws) == 0
    assert pkg.esc_convattn_last_path() == 6
    assert bool((buf[:1024] == 7.0).all()) and bool((buf[1024 + n:] == 7.0).all()), "write outside out"
    if mix:
        ref, mag = oracle.forward_pw(d["x"], C_a, d["w_large"], wp, d["w_dyn"], d["b_dyn"], want_mag=True)
    else:
        ref, mag = oracle.forward(d["x"], C_a, d["w_large"], d["w_dyn"], d["b_dyn"], want_mag=True)
    got = util.to_host_nchw(out, synth.NCHW)
    err = np.abs(got[:, :C_a] - ref[:, :C_a])
    bar = 2.0 ** -8 * np.abs(ref[:, :C_a]) * 1.001 + (2.0 ** -16 + 1e-5 if mix else 1e-5) * mag + 1e-30
    assert (err <= bar).all(), f"{int((err > bar).sum())} outputs beyond the bound, worst {(err / bar).max():.2f} bars"
    assert np.array_equal(got[:, C_a:], ref[:, C_a:])

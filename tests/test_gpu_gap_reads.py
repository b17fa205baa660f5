"""GPU parity of the pooling and dynamic-kernel stage (ESC paper, Eq. 4 lines 1-2) where its reads change: planes that do not
start on a 16-byte boundary, planes shorter than one piece, an odd number of channels for pairs of them, and the larger block
of maps from 1.5 M pixels on in each of its NHWC read modes.

Bar: fp32 sums of H*W values in any order and a dot product of C_a terms, 1e-5 of the sum of magnitudes."""
import numpy as np
import pytest

from paper_2503_06671_b200 import synth

pytestmark = pytest.mark.gpu

CASES = [
    # B, C, C_a, H, W
    (1, 5, 3, 1, 1), (2, 7, 5, 1, 3), (3, 9, 9, 3, 5), (2, 20, 7, 31, 33), (1, 16, 16, 180, 321), (4, 24, 1, 67, 9),
    (1, 9, 9, 1225, 1225), (1, 32, 16, 1224, 1226), (1, 24, 24, 1, 1500001), (301, 8, 8, 71, 71),
]


@pytest.mark.parametrize("layout", [synth.NCHW, synth.NHWC], ids=["nchw", "nhwc"])
@pytest.mark.parametrize("dtype", [synth.F32, synth.BF16], ids=["fp32", "bf16"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_dynamic_kernels(case, dtype, layout):
    import torch

    import paper_2503_06671_b200 as pkg

    B, C, C_a, H, W = case
    rng = np.random.default_rng(sum(case))
    g = torch.Generator(device="cuda").manual_seed(sum(case))
    x = torch.rand((B, C, H, W), generator=g, device="cuda") - 0.4 + torch.arange(C, device="cuda").view(1, C, 1, 1) / (2 * C)
    x = x.to(torch.bfloat16 if dtype == synth.BF16 else torch.float32)
    w, b = (synth.round_to(rng.uniform(-1, 1, s).astype(np.float32), dtype) for s in ((9 * C_a, C_a), (9 * C_a,)))
    mean = x[:, :C_a].double().mean((2, 3)).cpu().numpy()
    want = mean @ w.astype(np.float64).T + b
    bar = 1e-5 * (x[:, :C_a].double().abs().mean((2, 3)).cpu().numpy() @ np.abs(w).astype(np.float64).T + np.abs(b))
    xl = x if layout == synth.NCHW else x.permute(0, 2, 3, 1).contiguous()
    wt, bt = (torch.from_numpy(a).to("cuda", x.dtype) for a in (w, b))
    ws = pkg.new_workspace(B, C_a, H, W, 13)
    for _ in range(2):                                  # twice: the arrival counters start clean each launch
        dk = torch.full((B, C_a, 9), 7.0, device="cuda")
        pkg.esc_convattn_dynkernel(xl, C_a, wt, bt, dk, pkg.ESC_NCHW if layout == synth.NCHW else pkg.ESC_NHWC, ws)
        torch.cuda.synchronize()
        assert np.all(np.abs(dk.view(B, -1).double().cpu().numpy() - want) <= bar)

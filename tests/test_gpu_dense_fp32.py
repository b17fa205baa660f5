"""GPU parity for the dense large kernel (ESC paper, Section 3.2) on the FP32 pipe: the edges of its 64x8 tiles, every split
of the input channels over a cluster (1, 2, 4, 8 blocks: chosen by the number of tiles), and kernels smaller than the
compiled sizes (9, 13, 17).

Bars: fp32, 1e-5 of the sum of magnitudes, as for the other dense kernels; bf16, one rounding of the result beside it."""
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
    # B, C, H, W, K, dtype
    (1, 16, 8, 64, 13, synth.F32),       # one tile, nothing to copy through; eight blocks per cluster
    (2, 24, 9, 65, 13, synth.F32),       # one row and one column more
    (1, 64, 1, 1, 13, synth.F32),
    (1, 20, 7, 130, 3, synth.F32),       # 3x3: the middle of the 9x9 form
    (1, 32, 17, 20, 9, synth.F32),
    (1, 32, 23, 31, 11, synth.F32),      # in the 13x13 form
    (1, 48, 16, 70, 15, synth.F32),      # in the 17x17 form
    (1, 32, 30, 33, 17, synth.F32),
    (1, 32, 30, 33, 17, synth.BF16),     # bf16 with a kernel the tensor-core kernel does not take
    (592, 16, 5, 7, 13, synth.F32),      # 592 tiles: the input channels stay in one block
    (210, 16, 5, 7, 13, synth.F32),      # two blocks per cluster
    (450, 16, 5, 7, 13, synth.F32),      # four
]


@pytest.mark.parametrize("layout", [synth.NCHW, synth.NHWC])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_dense_fp32_pipe(pkg, oracle, case, layout):
    import torch

    B, C, H, W, K, dtype = case
    C_a = 16
    d = synth.make_inputs(B, C, C_a, H, W, K, dtype, seed=sum(case[:5]), per_image_scale=True, channel_means=True)
    wd = synth.make_dense_kernel(C_a, K, dtype, seed=sum(case[:5]))
    x = util.to_device(d["x"], dtype, layout)
    _, wdyn, bdyn = util.weights_to_device(d, dtype)
    n = x.numel()
    buf = torch.full((n + 2048,), 7.0, dtype=x.dtype, device="cuda")
    out = buf[1024:1024 + n].view(x.shape)
    ws = pkg.new_workspace(B, C_a, H, W, K)
    pkg.esc_convattn_forward_dense(x, C_a, K, torch.from_numpy(wd).to("cuda", util.torch_dtype(dtype)), wdyn, bdyn, out,
                                   util.layout_code(layout), ws)
    torch.cuda.synchronize()
    assert pkg.esc_convattn_device_status(ws) == 0
    assert bool((buf[:1024] == 7.0).all()) and bool((buf[1024 + n:] == 7.0).all()), "write outside out"
    ref, mag = oracle.forward_dense(d["x"], C_a, wd, d["w_dyn"], d["b_dyn"], want_mag=True)
    got = util.to_host_nchw(out, layout)
    err = np.abs(got[:, :C_a] - ref[:, :C_a])
    bar = 1e-5 * mag + 1e-30
    if dtype == synth.BF16:
        bar = bar + 2.0 ** -8 * np.abs(ref[:, :C_a]) * 1.001
    assert (err <= bar).all(), f"worst {(err / bar).max():.2f} bars"
    assert np.array_equal(got[:, C_a:], ref[:, C_a:])

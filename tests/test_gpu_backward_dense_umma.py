"""GPU parity for the gradient of the dense large kernel on the tcgen05 tensor cores (ESC paper, Section 3.2): the edges of its
units (strips of 16 to 64 columns, 8 to 32 rows), one to several units per block with the go tiles and the ring of input rows
re-used, and image changes inside a block, against the oracle's sums at sampled entries.

Bar: 1e-5 of the sum of magnitudes (exact bf16 products, fp32 accumulation), as for the warp-level kernel."""
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
    # B, C, H, W, K
    (1, 16, 1, 1, 13),         # one pixel
    (1, 24, 8, 16, 13),        # the smallest unit: 8 rows of 16 columns
    (2, 16, 9, 17, 13),        # one row and one column more
    (1, 32, 33, 65, 13),       # one more than the largest unit in both directions
    (3, 16, 40, 49, 9),        # K = 9: the middle of the sums
    (1, 16, 30, 130, 3),
    (40, 16, 96, 70, 13),      # 240 units: one or two per block, some of two images; both go tiles are used
    (7, 16, 400, 64, 13),      # seven rows of many units: the ring wraps several times inside a block
    (300, 16, 21, 19, 13),     # two or three small images per block: go tiles re-used
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_dense_weight_gradient(pkg, oracle, case):
    import torch

    B, C, H, W, K = case
    C_a = 16
    seed = sum(case)
    d = synth.make_inputs(B, C, C_a, H, W, K, synth.BF16, seed=seed, per_image_scale=True, channel_means=True)
    wdn = synth.make_dense_kernel(C_a, K, synth.BF16, seed=seed)
    go = synth.round_to(np.random.default_rng(seed).standard_normal(size=d["x"].shape).astype(np.float32), synth.BF16)
    x, god = util.to_device(d["x"], synth.BF16, synth.NHWC), util.to_device(go, synth.BF16, synth.NHWC)
    _, wd, bd = util.weights_to_device(d, synth.BF16)
    wdd = torch.from_numpy(wdn).to("cuda", torch.bfloat16)
    ws = pkg.new_backward_dense_workspace(B, C_a, H, W, K)
    got = []
    for _ in range(2):                                     # twice, bit for bit: fixed order of every sum
        g = torch.full((C_a, C_a, K, K), float("nan"), device="cuda")
        pkg.esc_convattn_backward_dense(x, god, C_a, K, wdd, wd, bd, torch.empty_like(x), g, None, None, pkg.ESC_NHWC, ws)
        torch.cuda.synchronize()
        assert pkg.esc_convattn_device_status(ws) == 0
        got.append(g.cpu().numpy())
    assert np.array_equal(got[0], got[1])
    idx = np.unique(np.concatenate([np.random.default_rng(seed + 1).integers(0, C_a * C_a * K * K, size=120),
                                    np.array([0, K * K - 1, C_a * C_a * K * K - 1, (5 * C_a + 5) * K * K + K * K // 2])]))
    vals, mags = oracle.backward_dense_points(d["x"], go, C_a, K, idx)
    err = np.abs(got[0].reshape(-1)[idx] - vals)
    assert (err <= 1e-5 * mags + 1e-30).all(), f"worst {(err / np.maximum(mags, 1e-30)).max():.3e} of its scale"

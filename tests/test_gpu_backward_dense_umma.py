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
    (7, 16, 400, 64, 13),      # 119 units of 24 rows, one per block: nine groups of input rows, one more than the ring holds
    (300, 16, 21, 19, 13),     # two or three small images per block, all of the same number of rows: go tiles re-used
]

# Three or more units per block, and the last segment of an image has fewer groups of four rows than the others: a go tile is used
# again after one that filled only part of it.
REUSE = [
    # B, C, H, W, K             segments of rows (groups of four)
    (64, 16, 73, 73, 13),      # 25, 25, 23 (7, 7, 6), two strips
    (4, 24, 361, 640, 13),     # eleven of 31 and one of 20 (8 and 5), ten strips
    (150, 16, 73, 50, 9),      # 25, 25, 23, one strip
]


@pytest.mark.parametrize("K", [3, 9, 11, 13])
@pytest.mark.parametrize("misaligned", [False, True])
def test_tcgen05_stencil_of_any_size_both_ways(pkg, oracle, K, misaligned):
    """The tcgen05 stencil kernel with a kernel smaller than 13x13 in the middle of zeros, weights that are not 16-byte aligned
    (staged another way), and the gradient's form (channels swapped, taps rotated, constants added): forward and grad_x, more
    rows per block than the ring and the row slots hold."""
    import torch

    B, C, C_a, H, W = 70, 24, 16, 45, 20
    d = synth.make_inputs(B, C, C_a, H, W, K, synth.BF16, seed=K, per_image_scale=True, channel_means=True)
    wdn = synth.make_dense_kernel(C_a, K, synth.BF16, seed=K)
    go = synth.round_to(np.random.default_rng(K).standard_normal(size=d["x"].shape).astype(np.float32), synth.BF16)
    x, god = util.to_device(d["x"], synth.BF16, synth.NHWC), util.to_device(go, synth.BF16, synth.NHWC)
    _, wd, bd = util.weights_to_device(d, synth.BF16)
    store = torch.zeros(wdn.size + 8, dtype=torch.bfloat16, device="cuda")
    wdd = store[1:1 + wdn.size] if misaligned else store[:wdn.size]
    wdd.copy_(torch.from_numpy(wdn).reshape(-1))
    wdd = wdd.view(wdn.shape)
    out, gx = torch.full_like(x, 7.0), torch.full_like(x, 7.0)
    ws = pkg.new_workspace(B, C_a, H, W, K)
    pkg.esc_convattn_forward_dense(x, C_a, K, wdd, wd, bd, out, pkg.ESC_NHWC, ws)
    assert pkg.esc_convattn_last_path() == 5
    wsb = pkg.new_backward_dense_workspace(B, C_a, H, W, K)
    pkg.esc_convattn_backward_dense(x, god, C_a, K, wdd, wd, bd, gx, None, None, None, pkg.ESC_NHWC, wsb)
    torch.cuda.synchronize()
    assert pkg.esc_convattn_device_status(ws) == 0 and pkg.esc_convattn_device_status(wsb) == 0
    ref, mag = oracle.forward_dense(d["x"], C_a, wdn, d["w_dyn"], d["b_dyn"], want_mag=True)
    got = util.to_host_nchw(out, synth.NHWC)
    err = np.abs(got[:, :C_a] - ref[:, :C_a])
    bar = 2.0 ** -8 * np.abs(ref[:, :C_a]) * 1.001 + 5e-5 * mag + 1e-30      # one rounding, tensor-core accumulation
    assert (err <= bar).all() and np.array_equal(got[:, C_a:], ref[:, C_a:])
    n = 6                                                   # images of the gradient that are compared
    rx = oracle.backward_dense(d["x"][:n], go[:n], C_a, wdn, d["w_dyn"], d["b_dyn"])[0]
    ax = oracle.backward_dense(np.abs(d["x"][:n]), np.abs(go[:n]), C_a, np.abs(wdn), np.abs(d["w_dyn"]), np.abs(d["b_dyn"]))[0]
    got = util.to_host_nchw(gx, synth.NHWC)[:n]
    err = np.abs(got[:, :C_a] - rx[:, :C_a])
    assert (err <= 2.0 ** -8 * np.abs(rx[:, :C_a]) * 1.001 + 5e-5 * ax[:, :C_a] + 1e-30).all()
    assert np.array_equal(got[:, C_a:], go[:n, C_a:].astype(np.float64))


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_dense_weight_gradient(pkg, oracle, case):
    _dense_weight_gradient(pkg, oracle, case, synth.NHWC)


@pytest.mark.parametrize("layout", [synth.NHWC, synth.NCHW])        # NCHW: the same kernel on packed tensors
@pytest.mark.parametrize("case", REUSE, ids=lambda c: "x".join(map(str, c)))
def test_dense_weight_gradient_unequal_segments(pkg, oracle, case, layout):
    _dense_weight_gradient(pkg, oracle, case, layout)


def _dense_weight_gradient(pkg, oracle, case, layout):
    import torch

    B, C, H, W, K = case
    C_a = 16
    seed = sum(case)
    d = synth.make_inputs(B, C, C_a, H, W, K, synth.BF16, seed=seed, per_image_scale=True, channel_means=True)
    wdn = synth.make_dense_kernel(C_a, K, synth.BF16, seed=seed)
    go = synth.round_to(np.random.default_rng(seed).standard_normal(size=d["x"].shape).astype(np.float32), synth.BF16)
    x, god = util.to_device(d["x"], synth.BF16, layout), util.to_device(go, synth.BF16, layout)
    _, wd, bd = util.weights_to_device(d, synth.BF16)
    wdd = torch.from_numpy(wdn).to("cuda", torch.bfloat16)
    ws = pkg.new_backward_dense_workspace(B, C_a, H, W, K)
    got = []
    for _ in range(2):                                     # twice, bit for bit: fixed order of every sum
        g = torch.full((C_a, C_a, K, K), float("nan"), device="cuda")
        pkg.esc_convattn_backward_dense(x, god, C_a, K, wdd, wd, bd, torch.empty_like(x), g, None, None, util.layout_code(layout), ws)
        torch.cuda.synchronize()
        assert pkg.esc_convattn_device_status(ws) == 0
        got.append(g.cpu().numpy())
    assert np.array_equal(got[0], got[1])
    idx = np.unique(np.concatenate([np.random.default_rng(seed + 1).integers(0, C_a * C_a * K * K, size=120),
                                    np.array([0, K * K - 1, C_a * C_a * K * K - 1, (5 * C_a + 5) * K * K + K * K // 2])]))
    vals, mags = oracle.backward_dense_points(d["x"], go, C_a, K, idx)
    err = np.abs(got[0].reshape(-1)[idx] - vals)
    assert (err <= 1e-5 * mags + 1e-30).all(), f"worst {(err / np.maximum(mags, 1e-30)).max():.3e} of its scale"

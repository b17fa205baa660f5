"""One workspace, zeroed once, serves calls of any shape in any order: every result must be, bit for bit, what a fresh workspace gives.
The shapes put dk and partial sums of one call where another counts arrivals, unless the counters have a place of their own; 700
images are more than that place holds.  Caller-owned workspaces, the library's own scratch and the host entry's slots."""
import pytest

from paper_2503_06671_b200 import synth
from tests import util

pytestmark = pytest.mark.gpu

C, C_A, K = 32, 16, 13
SHAPES = [(1, 360, 640), (64, 48, 48), (2, 100, 120), (1, 64, 64), (130, 24, 40), (700, 8, 24), (3, 90, 200), (64, 48, 48), (1, 360, 640),
          (700, 8, 24), (5, 64, 64)]
FORMS = [
    # entry, dtype, layout, large-kernel form, kernel size
    ("forward", synth.BF16, synth.NHWC, "depthwise", 13),      # one launch, the flags and counters of the images among CTAs
    ("forward", synth.BF16, synth.NCHW, "depthwise", 9),       # padded large kernel
    ("forward", synth.BF16, synth.NCHW, "dense", 13),          # packed map in the workspace
    ("forward", synth.F32, synth.NHWC, "depthwise", 13),       # two launches
    ("dynkernel", synth.BF16, synth.NHWC, "depthwise", 13),
    ("library", synth.F32, synth.NCHW, "depthwise", 13),
    ("host", synth.BF16, synth.NHWC, "depthwise", 13),
]


@pytest.mark.parametrize("case", FORMS, ids=lambda c: "-".join(map(str, c)))
def test_shapes_in_turn(case):
    import torch

    import paper_2503_06671_b200 as pkg

    entry, dtype, layout, form, K = case
    tdt, lay = util.torch_dtype(dtype), util.layout_code(layout)
    g = torch.Generator(device="cuda").manual_seed(1)

    def rand(*shape, scale=1.0):
        return (torch.randn(shape, generator=g, device="cuda") * scale).to(tdt)

    w_large = rand(C_A, C_A, K, K, scale=0.02) if form == "dense" else rand(C_A, K, K, scale=0.1)
    w_dyn, b_dyn = rand(9 * C_A, C_A, scale=0.25), rand(9 * C_A, scale=0.5)
    ws_of = {s: pkg.new_workspace(s[0], C_A, s[1], s[2], K) for s in set(SHAPES)}
    shared = torch.zeros(max(w.numel() for w in ws_of.values()), dtype=torch.uint8, device="cuda")

    def call(x, ws):
        B = x.shape[0]
        out = torch.empty((B, C_A, 3, 3), device="cuda") if entry == "dynkernel" else torch.full_like(x, 7.0)
        if entry == "dynkernel":
            pkg.esc_convattn_dynkernel(x, C_A, w_dyn, b_dyn, out, lay, ws)
        elif form == "dense":
            pkg.esc_convattn_forward_dense(x, C_A, K, w_large, w_dyn, b_dyn, out, lay, ws)
        else:
            pkg.esc_convattn_forward_ex(x, C_A, K, w_large, w_dyn, b_dyn, out, lay, ws)
        torch.cuda.synchronize()
        assert pkg.esc_convattn_device_status(ws) == 0
        return out

    for B, H, W in SHAPES:
        x = rand(*((B, H, W, C) if layout == synth.NHWC else (B, C, H, W)))
        x += torch.randn((B, 1, 1, 1), generator=g, device="cuda").to(tdt)
        want = call(x, pkg.new_workspace(B, C_A, H, W, K))
        for _ in range(2):
            if entry == "library":
                got = torch.full_like(x, 7.0)
                pkg.esc_convattn_forward(x, C_A, K, w_large, w_dyn, b_dyn, got)
                torch.cuda.synchronize()
            elif entry == "host":
                got = torch.empty_like(x, device="cpu", pin_memory=True)
                pkg.esc_convattn_forward_host(x.cpu().pin_memory(), C_A, K, *(t.cpu() for t in (w_large, w_dyn, b_dyn)), got, lay)
                got = got.cuda()
            else:
                got = call(x, shared)
            assert torch.equal(got, want), (B, H, W)


def test_first_use_while_the_default_stream_is_busy():
    """Scratch that the library allocates on a stream's first call is zero before the kernels count in it, also on a stream that does
    not wait for the default one."""
    import torch

    import paper_2503_06671_b200 as pkg

    B, H, W = 1, 640, 360
    x = torch.randn(B, C, H, W, device="cuda")
    ws = [torch.randn(s, device="cuda") * 0.1 for s in ((C_A, K, K), (9 * C_A, C_A), (9 * C_A,))]
    want, got = torch.empty_like(x), torch.empty_like(x)
    pkg.esc_convattn_forward_ex(x, C_A, K, *ws, want, pkg.ESC_NCHW, pkg.new_workspace(B, C_A, H, W, K))
    torch.cuda.synchronize()
    used = [torch.full((1 << 20,), -1, dtype=torch.int32, device="cuda") for _ in range(48)]     # what the driver hands out next
    torch.cuda.synchronize()
    del used
    torch.cuda.empty_cache()
    side = torch.cuda.Stream()
    torch.cuda._sleep(200_000_000)                          # about 0.1 s on the default stream
    pkg.esc_convattn_forward(x, C_A, K, *ws, got, stream=side)
    side.synchronize()
    assert torch.equal(got, want)

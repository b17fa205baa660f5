"""The host-buffer entries on NCHW tensors, whose identity channels travel beside the kernels in pieces in the blocking call: equal to
the device entry bit for bit, one and several images and pieces, both element types, odd widths, kernel sizes; two slots in turn."""
import pytest

from paper_2503_06671_b200 import synth

pytestmark = pytest.mark.gpu

CASES = [
    # B, C, C_a, H, W, K, dtype
    (1, 64, 16, 96, 120, 13, synth.BF16),      # one chunk, just large enough
    (2, 64, 16, 210, 333, 13, synth.BF16),     # images of 6.7 MB: two chunks each, the second one short; odd width
    (3, 48, 16, 77, 101, 9, synth.F32),
    (1, 40, 12, 250, 333, 17, synth.BF16),     # no tensor-core kernel takes it
    (1, 16, 16, 64, 64, 13, synth.F32),        # no identity channels
]


def _setup(case, seed):
    import torch

    B, C, C_a, H, W, K, dtype = case
    dt = torch.bfloat16 if dtype == synth.BF16 else torch.float32
    g = torch.Generator().manual_seed(seed)
    x = torch.randn((B, C, H, W), generator=g).to(dt).pin_memory()
    w = [(torch.randn(s, generator=g) / n).to(dt).pin_memory() for s, n in (((C_a, K, K), K), ((9 * C_a, C_a), C_a ** 0.5), ((9 * C_a,), 1))]
    return x, w


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_equals_device_entry(case):
    import torch

    import paper_2503_06671_b200 as pkg

    B, C, C_a, H, W, K, _ = case
    steps = []
    for seed in range(3):
        x, w = _setup(case, seed)
        out = torch.empty_like(x, device="cuda")
        pkg.esc_convattn_forward_ex(x.cuda(), C_a, K, *[t.cuda() for t in w], out, pkg.ESC_NCHW, pkg.new_workspace(B, C_a, H, W, K))
        steps.append((x, w, out.cpu(), torch.full_like(x, 7.0).pin_memory()))
    for i, (x, w, want, got) in enumerate(steps):
        pkg.esc_convattn_forward_host_submit(i % 2, x, C_a, K, *w, got, pkg.ESC_NCHW)
        if i > 0:
            pkg.esc_convattn_forward_host_wait((i - 1) % 2)
            assert torch.equal(steps[i - 1][3], steps[i - 1][2])
    pkg.esc_convattn_forward_host_wait((len(steps) - 1) % 2)
    assert torch.equal(steps[-1][3], steps[-1][2])
    x, w, want, got = steps[0]
    got.fill_(7.0)
    pkg.esc_convattn_forward_host(x, C_a, K, *w, got, pkg.ESC_NCHW)
    assert torch.equal(got, want)


# Batches whose images are smaller than a piece (several images a piece, the last piece with fewer), larger ones, and what must not
# overlap: pageable buffers, and an output that shares memory with the input.
MANY = [
    # B, C, C_a, H, W, K, dtype
    (23, 64, 16, 64, 64, 13, synth.BF16),      # ten images a piece: 10, 10, 3
    (40, 48, 16, 47, 53, 13, synth.BF16),      # images of 239 KB, odd planes
    (7, 24, 16, 64, 300, 9, synth.F32),        # 614 KB of identity channels an image: six and one
    (3, 64, 16, 210, 333, 13, synth.BF16),     # two pieces an image
]


@pytest.mark.parametrize("where", ["pinned", "pageable", "in_place", "shifted"])
@pytest.mark.parametrize("case", MANY, ids=lambda c: "x".join(map(str, c)))
def test_batches_and_buffers(case, where):
    import torch

    import paper_2503_06671_b200 as pkg

    B, C, C_a, H, W, K, dtype = case
    x, w = _setup(case, 11)
    want = torch.empty_like(x, device="cuda")
    pkg.esc_convattn_forward_ex(x.cuda(), C_a, K, *[t.cuda() for t in w], want, pkg.ESC_NCHW, pkg.new_workspace(B, C_a, H, W, K))
    want = want.cpu()
    n = x.numel()
    for _ in range(3):
        if where == "pinned":
            xi, got = x, torch.full_like(x, 7.0).pin_memory()
        elif where == "pageable":
            xi, got = x.clone(), torch.full_like(x, 7.0)
            assert not xi.is_pinned() and not got.is_pinned()
        else:                                                  # the input is read as a whole before anything comes back
            shift = 0 if where == "in_place" else C_a * H * W
            buf = torch.zeros(n + shift, dtype=x.dtype).pin_memory()
            xi, got = buf[shift:].view(x.shape), buf[:n].view(x.shape)
            xi.copy_(x)
        pkg.esc_convattn_forward_host(xi, C_a, K, *w, got, pkg.ESC_NCHW)
        assert torch.equal(got, want)

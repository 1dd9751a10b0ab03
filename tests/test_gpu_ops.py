"""The data-moving kernels of the surrogate (pooling, upsampling, their
adjoints, ReLU adjoint, BF16 cast, weight flip, sums of the weight gradient's
partials) where their access width changes: channel counts and row strides that
are and are not multiples of 8, bases off the 16-byte boundary, channel slices.
The references add in the kernels' order in FP32, so results are equal."""
import pytest

pytestmark = pytest.mark.gpu

# channels, row stride, channel offset: whole 16-byte rows, and ways to miss them
LAYOUTS = [(8, 8, 0), (32, 96, 64), (16, 24, 8), (8, 12, 0), (5, 7, 1), (24, 32, 4), (1, 1, 0), (40, 40, 0)]


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_1711_03254_gb300 import build
    build.build()
    from paper_1711_03254_gb300 import ws
    return torch, ws


def _view(torch, shape, layout, seed, dtype=None):
    c, ld, off = layout
    g = torch.Generator(device="cuda").manual_seed(seed)
    full = torch.randn(tuple(shape) + (ld,), generator=g, device="cuda").to(dtype or torch.bfloat16)
    return full, full[..., off:off + c]


def _children(t):
    return [t[:, a::2, b::2, d::2].float() for a in (0, 1) for b in (0, 1) for d in (0, 1)]


def _sum(parts):
    s = parts[0] * 0.0
    for p in parts:
        s = s + p
    return s


@pytest.mark.parametrize("layout", LAYOUTS, ids=str)
@pytest.mark.parametrize("accumulate", [False, True])
def test_resampling_and_relu(env, layout, accumulate):
    torch, ws = env
    c = layout[0]
    coarse, fine = (2, 3, 2, 5), (2, 6, 4, 10)
    _, x = _view(torch, fine, layout, 1)
    _, y = _view(torch, coarse, layout, 2)
    keep, p = _view(torch, coarse, layout, 3)
    before = keep.clone()
    ws.ws_avgpool2(x, p)
    assert torch.equal(p, (_sum(_children(x)) * 0.125).to(torch.bfloat16))
    off = layout[2]
    before[..., off:off + c] = p
    assert torch.equal(keep, before)  # nothing outside the slice is written
    _, u = _view(torch, fine, layout, 4)
    ws.ws_upsample2(y, u)
    up = y.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)
    assert torch.equal(u, up)
    _, dx = _view(torch, fine, layout, 5)
    want = up.float() * 0.125 + (dx.float() if accumulate else 0.0)
    ws.ws_avgpool2_bwd(y, dx, accumulate=accumulate)
    assert torch.equal(dx, want.to(torch.bfloat16))
    _, dc = _view(torch, coarse, layout, 6)
    want = _sum(_children(x)) + (dc.float() if accumulate else 0.0)
    ws.ws_upsample2_bwd(x, dc, accumulate=accumulate)
    assert torch.equal(dc, want.to(torch.bfloat16))
    _, act = _view(torch, fine, layout, 7)
    act[0, 0, 0, 0, 0] = float("nan")
    act[0, 0, 0, 1, 0] = 0.0
    _, g = _view(torch, fine, layout, 8)
    want = torch.where(act.float() > 0.0, g, torch.zeros_like(g))
    ws.ws_relu_bwd(act, g)
    assert torch.equal(g, want)
    _, f = _view(torch, fine, layout, 9, torch.float32)
    _, b = _view(torch, fine, layout, 10)
    ws.ws_to_bf16(f, b)
    assert torch.equal(b, f.to(torch.bfloat16))


@pytest.mark.parametrize("co,ci,k", [(16, 16, 3), (48, 80, 3), (64, 160, 1), (33, 5, 3), (1, 1, 1)])
def test_flip_weights(env, co, ci, k):
    torch, ws = env
    w = torch.randn((co, k, k, k, ci), device="cuda").to(torch.bfloat16)
    wf = torch.empty((ci, k, k, k, co), dtype=torch.bfloat16, device="cuda")
    ws.ws_conv3d_flip_weights(w, wf)
    assert torch.equal(wf, w.flip(1, 2, 3).permute(4, 1, 2, 3, 0))

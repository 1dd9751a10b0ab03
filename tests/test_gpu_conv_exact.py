"""Convolutions of small whole numbers, whose sums FP32 holds exactly in any order
(at most 2^24): the results equal the integer ones.  Covers both block shapes of the
partial sums of the weight gradient (4 and 8 rows) on either side of their line, with
and without a bias gradient, for resident and gathered partials."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_1711_03254_gb300 import build
    build.build()
    from paper_1711_03254_gb300 import ws
    return torch, ws


def _ints(torch, shape, seed, lo=-3, hi=4):
    return torch.randint(lo, hi, shape, generator=torch.Generator().manual_seed(seed)).cuda()


def _wgrad(torch, x, dy, k):
    """dW [Co, k, k, k, Ci] and db in 64-bit integers' exact FP64."""
    N, D, H, W, Ci = x.shape
    r = k // 2
    xp = torch.nn.functional.pad(x.double(), (0, 0, r, r, r, r, r, r))
    g = dy.double().reshape(-1, dy.shape[-1])
    dw = torch.empty((dy.shape[-1], k, k, k, Ci), dtype=torch.float64, device="cuda")
    for a in range(k):
        for b in range(k):
            for c in range(k):
                dw[:, a, b, c] = g.T @ xp[:, a:a + D, b:b + H, c:c + W].reshape(-1, Ci)
    return dw, g.sum(0)


@pytest.mark.parametrize("Ci,Co,k", [(16, 16, 3), (32, 48, 3), (96, 32, 3), (80, 48, 3), (64, 64, 3), (48, 160, 3),
                                     (16, 16, 1), (160, 64, 1), (224, 256, 1)])
@pytest.mark.parametrize("shape", [(2, 5, 7, 9), (1, 9, 33, 30), (1, 2, 3, 260)])
@pytest.mark.parametrize("bias", [True, False])
def test_weight_gradient_sums_are_exact(env, shape, Ci, Co, k, bias):
    torch, ws = env
    x, dy = _ints(torch, shape + (Ci,), Ci), _ints(torch, shape + (Co,), Co + 1)
    want, want_b = _wgrad(torch, x, dy, k)
    assert float(want.abs().max()) < 2 ** 24
    dw, db = torch.ones(want.shape, device="cuda"), torch.ones(Co, device="cuda")
    ws.ws_conv3d_bwd_weight(x.to(torch.bfloat16), dy.to(torch.bfloat16), dw, db if bias else None, k)
    assert ws.ws_tc_status() == 0
    assert torch.equal(dw.double(), want + 1.0)
    assert torch.equal(db.double(), want_b + 1.0 if bias else torch.ones_like(want_b))


@pytest.mark.parametrize("Ci,Co,k", [(16, 16, 3), (48, 32, 3), (16, 256, 3), (32, 112, 3), (80, 48, 1), (16, 160, 1)])
@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (1, 2, 3, 260), (2, 3, 5, 7)])
@pytest.mark.parametrize("f32", [True, False])
def test_gathered_forward_is_exact(env, shape, Ci, Co, k, f32):
    """The gathered kernel (lines wider than 254, wide 1x1x1, or on request) with and without
    bias and ReLU; in BF16 the rounded exact result."""
    torch, ws = env
    x, w, b = _ints(torch, shape + (Ci,), Ci), _ints(torch, (Co, k, k, k, Ci), Co), _ints(torch, (Co,), 9, -50, 50)
    r = k // 2
    xp = torch.nn.functional.pad(x.double(), (0, 0, r, r, r, r, r, r))
    N, D, H, W = shape
    y = sum(xp[:, i:i + D, j:j + H, l:l + W] @ w[:, i, j, l].double().T
            for i in range(k) for j in range(k) for l in range(k))
    assert float(y.abs().max()) + 50 < 2 ** 24
    prev = ws.ws_conv3d_fwd_algo("gather")
    try:
        for bias, relu in ((b.float(), True), (None, False), (b.float(), False)):
            out = torch.full(shape + (Co + 8,), 3.0, dtype=torch.float32 if f32 else torch.bfloat16, device="cuda")
            ws.ws_conv3d_fwd(x.to(torch.bfloat16), w.to(torch.bfloat16), bias, out[..., :Co], relu)
            want = y + (b.double() if bias is not None else 0.0)
            want = (want.clamp(min=0.0) if relu else want).to(out.dtype)
            assert torch.equal(out[..., :Co], want) and bool((out[..., Co:] == 3.0).all())
    finally:
        ws.ws_conv3d_fwd_algo(prev)
    assert ws.ws_tc_status() == 0

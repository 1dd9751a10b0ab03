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

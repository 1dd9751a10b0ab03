"""Host-side plans of the automatic choice (no GPU needed): forward grids that are
split over fewer lines or over the output channels, and the weight gradient with
three copies of dY.  As for the other plans, they must stay inside the limits the
kernels rely on, for devices of several SM counts, and a replay of the tiling with
the returned plan must give the direct correlation."""
import itertools
import math

import numpy as np
import pytest

from .test_conv_plans import (SHAPES, SMEM_PER_BLOCK, _direct, _direct_wgrad, _replay_forward, _resident_per_sm, algos,
                              ws)  # noqa: F401

SMS = [1, 13, 152]


@pytest.mark.parametrize("sms", SMS)
def test_automatic_forward_plans_stay_within_limits(ws, algos, sms):  # noqa: F811
    split = fewer = 0
    for (N, D, H, W), Ci, Co in itertools.product(SHAPES, (16, 32, 96, 224), (16, 32, 64, 96, 128, 160, 256)):
        ws.ws_conv3d_fwd_algo("resident")
        whole = ws.ws_conv3d_plan_for(sms, "fwd", N, D, H, W, Ci, Co)
        ws.ws_conv3d_fwd_algo("auto")
        p = ws.ws_conv3d_plan_for(sms, "fwd", N, D, H, W, Ci, Co)
        assert whole["nco"] == 1 and not whole["persistent"]
        assert Co % (16 * p["nco"]) == 0 and not p["persistent"] and p["buf_cols"] == 0
        n = Co // p["nco"]  # output channels of a block
        pitch, by, rows = p["pitch"], p["by"], p["a_half"] // 16
        assert pitch == W + 2 <= 256 and 1 <= by <= H and by + 2 <= 256 and p["nyt"] == math.ceil(H / by)
        assert p["ntiles"] == math.ceil(((by - 1) * pitch + W) / 128)
        assert (by + 2) * pitch <= rows and 128 * p["ntiles"] - 1 + 2 * pitch + 2 < rows
        # the input tile and every tap's weights start on the 256 bytes the swizzle repeats after
        assert 2 * p["a_half"] % 256 == 0 and 32 * n % 256 == 0 and p["stage_bytes"] % 256 == 0
        assert p["stage_bytes"] == 2 * p["a_half"] + 9 * n * 32
        assert p["tx_bytes"] == (by + 2) * pitch * 32 + 9 * n * 32 < 1 << 20
        assert p["stages"] >= 2 and p["smem"] <= SMEM_PER_BLOCK and Co * 4 <= p["stage_bytes"]  # (bias in stage 0)
        assert 1023 + p["stages"] * p["stage_bytes"] + 8 * (2 * p["stages"] + 1) + 8 <= p["smem"]
        assert p["stages"] * p["stage_bytes"] + 1024 <= 256 * 1024
        assert p["cols"] in (32, 64, 128, 256, 512) and p["ntiles"] * n <= p["cols"]
        assert _resident_per_sm(p["smem"]) * p["cols"] <= 512 and p["per_sm"] * p["cols"] <= 512
        assert p["grid"] == N * D * p["nyt"] * p["nco"]
        split += p["nco"] > 1
        fewer += p["by"] < whole["by"]
    if sms > 1:
        assert split > 100 and fewer > 100  # both ways of splitting are among the plans


def _parts(p, w):
    """The blocks' weights: nco runs of output channels."""
    n = w.shape[0] // p["nco"]
    return [w[i * n:(i + 1) * n] for i in range(p["nco"])]


@pytest.mark.parametrize("sms", SMS)
@pytest.mark.parametrize("shape,Ci,Co", [((1, 3, 9, 12), 32, 96), ((2, 2, 5, 7), 16, 48), ((1, 2, 7, 40), 32, 64),
                                         ((1, 8, 8, 8), 32, 128), ((1, 4, 16, 16), 16, 160), ((1, 1, 1, 1), 16, 256)])
def test_automatic_forward_tiling_replays_the_correlation(ws, algos, sms, shape, Ci, Co):  # noqa: F811
    ws.ws_conv3d_fwd_algo("auto")
    rng = np.random.default_rng(sum(shape) + Ci + Co)
    x = rng.standard_normal(shape + (Ci,))
    w = rng.standard_normal((Co, 27, Ci))
    p = ws.ws_conv3d_plan_for(sms, "fwd", *shape, Ci, Co)
    y = np.concatenate([_replay_forward(x, part, p) for part in _parts(p, w)], axis=-1)
    ref = _direct(x, w)
    assert y.shape == ref.shape and not np.isnan(y).any()
    assert np.abs(y - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("sms", SMS)
def test_weight_gradient_plans_with_copies_stay_within_limits(ws, algos, sms):  # noqa: F811
    ws.ws_conv3d_bwd_weight_algo("auto")
    planned = 0
    for (N, D, H, W), Ci, Co in itertools.product(SHAPES, (16, 32, 64, 96, 128), (16, 32, 48, 64, 160)):
        p = ws.ws_conv3d_plan_for(sms, "wgrad", N, D, H, W, Ci, Co)
        if p is None or p["dz"] != 2:
            # tap pairs or gathered rows, unless the copies' two stages of one line do not fit
            ks = math.ceil((W + 2) / 16)
            rows = (max(3 * (W + 2), ks * 16 + 2 * (W + 2)) + 7) // 8 * 8
            stage = max(6 * rows * 32 + (1 + 3 * Co // 16) * ks * 512, 8 * rows * 32)
            assert Ci % 32 or Co > 48 or 2 * stage + 1024 + 64 > SMEM_PER_BLOCK, (N, D, H, W, Ci, Co)
            continue
        planned += 1
        assert Ci % 32 == 0 and Co <= 48 and p["ci_blk"] == 32 and p["grid_y"] == Ci // 32
        pitch, by, ks = p["pitch"], p["by"], p["ksteps"]
        gx, gy = 2 * p["region"], ks * 512  # bytes of a 16-channel group of X and of dY
        assert pitch == W + 2 <= 256 and 1 <= by <= H and by + 2 <= 256 and ks == math.ceil(by * pitch / 16)
        assert gx % 256 == 0 and p["stage_bytes"] % 256 == 0
        # X boxes, and the rows the dy shifts reach, within a group; dY boxes within theirs
        assert (by + 2) * pitch * 32 <= gx and (ks * 16 + 2 * pitch) * 32 <= gx and by * pitch * 32 <= gy
        # six X groups, the ones, three copies of dY; the eighth M group is read and dropped
        assert p["stage_bytes"] >= 6 * gx + gy + 3 * (Co // 16) * gy and p["stage_bytes"] >= 8 * gx
        assert 9 * Co <= p["cols"] <= 512 and 3 * Co <= 256 and 3 * Co % 16 == 0
        assert (6 * (by + 2) + 3 * (Co // 16) * by) * pitch * 32 < 1 << 20
        assert p["stages"] >= 2 and p["smem"] <= SMEM_PER_BLOCK
        assert 1023 + p["stages"] * p["stage_bytes"] + 8 * (2 * p["stages"] + 1) + 8 <= p["smem"]
        assert _resident_per_sm(p["smem"]) * p["cols"] <= 512
        nkb = N * D * p["nyb"]
        assert p["nyb"] == math.ceil(H / by) and p["npb"] * p["kpb"] >= nkb > (p["npb"] - 1) * p["kpb"]
    assert planned > 300


def _box16(t, c0, x0, y0, z, n, pitch, lines):
    """A TMA box of 16 channels: rows (line, column) from (x0, y0) of plane z, zeros outside."""
    N, D, H, W, C = t.shape
    out = np.zeros((lines, pitch, 16))
    if 0 <= z < D:
        ys, xs = y0 + np.arange(lines), x0 + np.arange(pitch)
        vy, vx = (ys >= 0) & (ys < H), (xs >= 0) & (xs < W)
        out[np.ix_(vy, vx)] = t[n, z][np.ix_(ys[vy], xs[vx])][..., c0:c0 + 16]
    return out.reshape(lines * pitch, 16)


def _replay_copies(x, dy, p, left=1):
    """The weight gradient with three copies of dY, on a stage of 32-byte rows (16 channels):
    groups (dz, 16 channels) of X, the ones, then groups (copy dx, 16 channels) of dY loaded
    dx columns to the left (`left`: columns per copy, 1).  Per K-step and dy one product of
    M = 8 groups, one X group apart, with N = 3 Co; what a K-block's loads do not cover keeps
    its earlier contents.  Returns (dW [Co, 27, Ci], db [Co])."""
    N, D, H, W, Ci = x.shape
    Co = dy.shape[-1]
    pitch, by, ks = p["pitch"], p["by"], p["ksteps"]
    gx, gy, nb, rows = p["region"] // 16, ks * 16, Co // 16, p["stage_bytes"] // 32
    y_off = 6 * gx + gy
    nkb = N * D * p["nyb"]
    dw, db = np.zeros((Co, 27, Ci)), np.zeros(Co)
    for pb, cb in itertools.product(range(p["npb"]), range(Ci // 32)):
        sm = np.zeros((rows, 16))
        if cb == 0:
            sm[6 * gx:y_off] = 1.0
        acc = np.zeros((3, 128, 3 * Co))
        for kb in range(pb * p["kpb"], min((pb + 1) * p["kpb"], nkb)):
            yb, z, n = kb % p["nyb"], (kb // p["nyb"]) % D, kb // (p["nyb"] * D)
            y0 = yb * by
            for dz, g in itertools.product(range(3), range(2)):
                at = (dz * 2 + g) * gx
                sm[at:at + (by + 2) * pitch] = _box16(x, cb * 32 + 16 * g, -1, y0 - 1, z + dz - 1, n, pitch, by + 2)
            for dx, g in itertools.product(range(3), range(nb)):
                at = y_off + (dx * nb + g) * gy
                sm[at:at + by * pitch] = _box16(dy, 16 * g, -dx * left, y0, z, n, pitch, by)
            for k, dyy in itertools.product(range(ks), range(3)):
                a0, b0 = 16 * k + dyy * pitch, y_off + 16 * k
                assert 7 * gx + a0 + 16 <= rows and b0 + (3 * nb - 1) * gy + 16 <= rows
                a = np.concatenate([sm[m * gx + a0:m * gx + a0 + 16] for m in range(8)], axis=1)
                b = np.concatenate([sm[b0 + j * gy:b0 + j * gy + 16] for j in range(3 * nb)], axis=1)
                acc[dyy] += a.T @ b
        for dz, dyy, dx in itertools.product(range(3), range(3), range(3)):
            dw[:, dz * 9 + dyy * 3 + dx, cb * 32:cb * 32 + 32] += acc[dyy, dz * 32:dz * 32 + 32,
                                                                      dx * Co:(dx + 1) * Co].T
        if cb == 0:
            db += acc[0, 96, :Co]
    return dw, db


@pytest.mark.parametrize("shape,Ci,Co", [((1, 3, 6, 12), 32, 32), ((2, 2, 5, 9), 64, 48), ((1, 2, 4, 7), 96, 16),
                                         ((1, 1, 1, 1), 32, 16), ((1, 2, 3, 130), 32, 16), ((1, 1, 70, 3), 32, 16)])
def test_weight_gradient_with_copies_replays_the_correlation(ws, algos, shape, Ci, Co):  # noqa: F811
    ws.ws_conv3d_bwd_weight_algo("auto")
    rng = np.random.default_rng(sum(shape) + Ci + Co)
    x = rng.standard_normal(shape + (Ci,))
    dy = rng.standard_normal(shape + (Co,))
    p = ws.ws_conv3d_plan_for(3, "wgrad", *shape, Ci, Co)
    assert p["dz"] == 2
    dw, db = _replay_copies(x, dy, p)
    ref, ref_b = _direct_wgrad(x, dy), dy.reshape(-1, Co).sum(axis=0)
    assert np.abs(dw - ref).max() <= 1e-12 * np.abs(ref).max()
    assert np.abs(db - ref_b).max() <= 1e-12 * np.abs(ref_b).max()


def test_copies_replay_catches_a_wrong_shift(ws, algos):  # noqa: F811
    """Copies of dY two columns apart instead of one must not pass."""
    rng = np.random.default_rng(4)
    x, dy = rng.standard_normal((1, 2, 4, 7, 32)), rng.standard_normal((1, 2, 4, 7, 16))
    ws.ws_conv3d_bwd_weight_algo("auto")
    p = ws.ws_conv3d_plan_for(1, "wgrad", 1, 2, 4, 7, 32, 16)
    dw, _ = _replay_copies(x, dy, p, left=2)
    assert np.abs(dw - _direct_wgrad(x, dy)).max() > 1e-3

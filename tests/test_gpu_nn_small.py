"""The surrogate's reduction and packing kernels at the sizes where their loops end
(single pixels, group and block remainders), for buffers on and off 16-byte
boundaries, and for values outside the float range of the loss's fast form."""
import ctypes

import numpy as np
import pytest

from paper_2402_15752_gb300 import surrogate as sg

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24


def _t():
    import torch
    return torch


def _p(t):
    return None if t is None else ctypes.c_void_p(t.data_ptr())


def _s():
    return ctypes.c_void_p(_t().cuda.current_stream().cuda_stream)


def _dev(a, shift, dtype=None):
    """`a` on the device, its first element `shift` elements into an allocation."""
    t = _t()
    src = t.from_numpy(np.ascontiguousarray(a))
    src = src if dtype is None else src.to(dtype)
    buf = t.zeros(src.numel() + shift, dtype=src.dtype, device="cuda")
    v = buf[shift:].view(src.shape)
    v.copy_(src)
    return v


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("co", [16, 48])
@pytest.mark.parametrize("P", [1, 41, 128, 43 * 1024 * 4 + 7])
def test_bias_gradient(P, co, shift):
    t = _t()
    x = np.random.default_rng(P + co).standard_normal((P, co)).astype(np.float32)
    dy = _dev(x, shift, t.bfloat16)
    db = t.empty(co, device="cuda")
    part = t.empty(1024 * co, device="cuda")
    assert sg.nn_lib().lbm_nn_bias_grad(_p(dy), co, P, _p(db), _p(part), _s()) == 0
    ref = dy.double().cpu().numpy()
    # additions along one output: a thread's pixels, its block's threads, the blocks' tree
    adds = P / (1024 * 128 / (co / 16) / 3) + 128 + 4 + 8 + 2
    np.testing.assert_array_less(np.abs(db.cpu().numpy() - ref.sum(0)), adds * EPS * np.abs(ref).sum(0) + 1e-30)


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("used", [1, 5, 16])
@pytest.mark.parametrize("P", [1, 255, 257, 1024 * 256 + 3])
def test_loss_and_its_gradient(P, used, shift):
    t = _t()
    g = np.random.default_rng(P + used)
    pred = g.standard_normal((P, 16)).astype(np.float32)
    targ = (pred + g.standard_normal((P, 16)) * 10.0 ** g.uniform(-6, 2, (P, 16))).astype(np.float32)
    _check_loss(t, pred, targ, used, shift)


@pytest.mark.parametrize("big", [3e19, 1e-20, 0.0])
def test_loss_outside_the_float_range(big):
    t = _t()
    g = np.random.default_rng(3)
    pred = g.standard_normal((300, 16)).astype(np.float32)
    targ = g.standard_normal((300, 16)).astype(np.float32)
    pred[7, 2], targ[7, 2] = big, -big
    pred[8, 1], targ[8, 1] = big, 0.0
    _check_loss(t, pred, targ, 5, 0)


def test_loss_of_tiny_differences_only_and_of_nan():
    t = _t()
    pred = np.full((65, 16), 1e-22, np.float32)
    _check_loss(t, pred, np.zeros_like(pred), 5, 0)
    pred[3, 4] = np.nan
    loss, _ = _loss(t, pred, np.zeros_like(pred), 5, 0)
    assert np.isnan(loss)
    pred[3, 4] = np.inf
    loss, _ = _loss(t, pred, np.zeros_like(pred), 5, 0)
    assert np.isinf(loss)


def _loss(t, pred, targ, used, shift):
    P = pred.shape[0]
    part = t.empty(1024, dtype=t.float64, device="cuda")
    loss = t.zeros(1, dtype=t.float64, device="cuda")
    dz = _dev(np.ones((P, 16), np.float32), shift, t.bfloat16)
    assert sg.nn_lib().lbm_nn_mse(_p(_dev(pred, shift)), _p(_dev(targ, shift)), used, P, _p(dz), _p(part), _p(loss),
                                  _s()) == 0
    return float(loss.item()), dz.double().cpu().numpy()


def _check_loss(t, pred, targ, used, shift):
    P = pred.shape[0]
    loss, dz = _loss(t, pred, targ, used, shift)
    d = pred[:, :used].astype(np.float64) - targ[:, :used].astype(np.float64)
    # sums of positive terms: 2^-44 per pixel's pair, 2^-53 per addition in double
    assert loss == pytest.approx(float((d ** 2).sum() / (P * used)), rel=1e-12, abs=0.0)
    # the double product rounded to float and then to bfloat16, bit for bit
    want = np.zeros((P, 16), np.float32)
    want[:, :used] = (2.0 * (1.0 / (float(P) * used)) * d).astype(np.float32)
    np.testing.assert_array_equal(dz, t.from_numpy(want).to(t.bfloat16).double().numpy())


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("B,H,W", [(1, 1, 1), (2, 1, 31), (3, 3, 11), (2, 16, 16), (5, 40, 333)])
def test_pack_and_unpack(B, H, W, shift):
    t = _t()
    g = np.random.default_rng(B * H * W)
    f = g.standard_normal((B, 6, H, W)).astype(np.float32)
    sh, sc = g.standard_normal(5).astype(np.float32), g.uniform(0.5, 2.0, 5).astype(np.float32)
    fd, shd, scd = (t.from_numpy(a).cuda() for a in (f, sh, sc))
    state = _dev(np.full((B, H, W, 16), np.nan, np.float32), shift)
    act = _dev(np.full((B, H, W, 16), np.nan, np.float32), shift, t.bfloat16)
    L = sg.nn_lib()
    assert L.lbm_nn_pack(_p(fd), B, H, W, _p(shd), _p(scd), _p(state), _p(act), _s()) == 0
    v = np.stack([f[:, 0], f[:, 1], f[:, 2], f[:, 3], f[:, 4] + f[:, 5]], -1)
    want = np.zeros((B, H, W, 16), np.float32)
    want[..., :5] = (v - sh) * sc
    np.testing.assert_array_equal(state.cpu().numpy(), want)
    assert t.equal(act.cpu(), t.from_numpy(want).to(t.bfloat16))
    out = t.full((B, 5, H, W), float("nan"), device="cuda")
    assert L.lbm_nn_unpack(_p(state), B, H, W, _p(shd), _p(scd), _p(out), _s()) == 0
    np.testing.assert_array_equal(out.cpu().numpy(), np.moveaxis(want[..., :5] / sc + sh, -1, 1))

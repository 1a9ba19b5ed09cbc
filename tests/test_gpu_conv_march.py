"""The convolution kernels where their rings wrap and their runs cross strips: CTAs
that march down many rows, runs of one or two rows, single-row strips, every dilation
class, against the same sums in plain 64-bit torch."""
import ctypes

import pytest

from paper_2402_15752_gb300 import surrogate as sg

pytestmark = pytest.mark.gpu

U_BF16 = 2.0 ** -8
ACC = 1e-5  # FP32 accumulation, relative to the sum of |terms|


def _p(t):
    return None if t is None else ctypes.c_void_p(t.data_ptr())


def _conv(torch, x, w, d):
    out = 0.0
    for t in range(9):
        out = out + torch.roll(x, (-(t // 3 - 1) * d, -(t % 3 - 1) * d), (1, 2)) @ w[:, t].T
    return out


def _wgrad(torch, x, dy, d):
    return torch.stack([dy.flatten(0, 2).T @ torch.roll(x, (-(t // 3 - 1) * d, -(t % 3 - 1) * d), (1, 2)).flatten(0, 2)
                        for t in range(9)], 1)


# rows per CTA (of 152): 20.2, 20.2, 10.5 (rings wrap, runs cross strips), 1 and 2 (short
# runs), single-row strips, an odd count
SHAPES = [(2, 768, 256, 1), (2, 768, 256, 8), (8, 200, 128, 4), (1, 8, 128, 8), (3, 62, 128, 2), (1, 7, 256, 1)]


@pytest.mark.parametrize("B,H,W,d", SHAPES)
@pytest.mark.parametrize("ci,co", [(16, 48), (48, 48), (48, 16)])
def test_convolution_and_weight_gradient(ci, co, B, H, W, d):
    import torch
    L = sg.nn_lib()
    g = torch.Generator(device="cuda").manual_seed(B * H + d)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    x, dy = rnd(B, H, W, ci).to(torch.bfloat16), rnd(B, H, W, co).to(torch.bfloat16)
    w, b, res = rnd(co, 9, ci).to(torch.bfloat16), rnd(co), rnd(B, H, W, co)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    want = _conv(torch, x.double(), w.double(), d) + b.double()
    size = _conv(torch, x.double().abs(), w.double().abs(), d) + b.double().abs()
    if co == 48:
        y = torch.full((B, H, W, co), float("nan"), dtype=torch.bfloat16, device="cuda")
        assert L.lbm_nn_conv3x3(_p(x), ci, _p(w), _p(b), co, sg.RELU, None, None, _p(y), B, H, W, d, _p(st), s) == 0
        want = want.clamp(min=0)
        assert bool(((y.double() - want).abs() <= ACC * size + U_BF16 * want.abs()).all())
        mask = rnd(B, H, W, co).to(torch.bfloat16)
        y.fill_(float("nan"))
        assert L.lbm_nn_conv3x3(_p(x), ci, _p(w), None, co, sg.MASK, None, _p(mask), _p(y), B, H, W, d, _p(st), s) == 0
        want = _conv(torch, x.double(), w.double(), d) * (mask > 0)
        assert bool(((y.double() - want).abs() <= ACC * size + U_BF16 * want.abs()).all())
    else:
        want = want + res.double()
        y = res.clone()  # in place, as the two-hop gradient uses it
        assert L.lbm_nn_conv3x3(_p(x), ci, _p(w), _p(b), co, sg.RESIDUAL, _p(y), None, _p(y), B, H, W, d, _p(st), s) == 0
        assert bool(((y.double() - want).abs() <= ACC * (size + res.double().abs())).all())
    nb = L.lbm_nn_wgrad_partial_bytes(ci, co, B, H, W, d)
    part = torch.full((nb // 4,), float("nan"), device="cuda")
    dw = torch.full((co, 9, ci), float("nan"), device="cuda")
    assert L.lbm_nn_conv3x3_wgrad(_p(x), ci, _p(dy), co, _p(dw), _p(part), nb, B, H, W, d, _p(st), s) == 0
    want = _wgrad(torch, x.double(), dy.double(), d)
    size = _wgrad(torch, x.double().abs(), dy.double().abs(), d)
    assert bool(((dw.double() - want).abs() <= ACC * size).all())
    # with the bias gradient: the same weight gradient, bit for bit
    dw2, db = torch.full_like(dw, float("nan")), torch.full((co,), float("nan"), device="cuda")
    bpart = torch.full((nb // (36 * ci),), float("nan"), device="cuda")
    assert L.lbm_nn_conv3x3_wgrad_bias(_p(x), ci, _p(dy), co, _p(dw2), _p(db), _p(part), nb, _p(bpart), B, H, W, d,
                                       _p(st), s) == 0
    assert torch.equal(dw, dw2)
    assert bool(((db.double() - dy.double().sum((0, 1, 2))).abs() <= ACC * dy.double().abs().sum((0, 1, 2))).all())
    assert int(st.item()) == 0

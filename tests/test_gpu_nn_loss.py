"""The loss carries double precision: against the exact rational sum of squares.

One pixel: its squares are summed to better than 2^-60, rounded twice on the way into a
double and twice more by the factor 1 / (pixels x channels): 4 roundings of 2^-53, and one
unit to spare.  More pixels add one rounding per addition along a sum."""
import ctypes
from fractions import Fraction

import numpy as np
import pytest

from paper_2402_15752_gb300 import surrogate as sg

pytestmark = pytest.mark.gpu


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def _loss(pred, targ, used):
    import torch
    P = pred.shape[0]
    a, b = torch.from_numpy(pred).cuda(), torch.from_numpy(targ).cuda()
    part = torch.empty(1024, dtype=torch.float64, device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert sg.nn_lib().lbm_nn_mse(_p(a), _p(b), used, P, None, _p(part), _p(loss), s) == 0
    return float(loss.item())


def _exact(pred, targ, used):
    t = Fraction(0)
    for x, y in zip(pred[:, :used].ravel(), targ[:, :used].ravel()):
        d = Fraction(float(x)) - Fraction(float(y))
        t += d * d
    return t / (pred.shape[0] * used)


@pytest.mark.parametrize("used", [1, 3, 5, 8, 11, 16])
@pytest.mark.parametrize("spread", [0.0, 3.0])
@pytest.mark.parametrize("P", [1, 600])
def test_the_loss_has_the_bits_of_a_double(P, spread, used):
    g = np.random.default_rng(100 * used + int(spread) + P)
    # the additions of a pixel's sum to others: a thread's, its warp's 5, the block's 8, the blocks' tree of 8
    roundings = 5 if P == 1 else 5 + 2 + 5 + 8 + 8
    for _ in range(40 if P == 1 else 4):
        pred = (g.standard_normal((P, 16)) * 10.0 ** g.uniform(-spread, spread, (P, 16))).astype(np.float32)
        targ = (pred * g.uniform(0, 1) + g.standard_normal((P, 16)) * 10.0 ** g.uniform(-2 * spread, 0, (P, 16))).astype(
            np.float32)
        want = _exact(pred, targ, used)
        err = abs(Fraction(_loss(pred, targ, used)) - want) / want
        assert err <= Fraction(roundings, 2 ** 53), float(err * 2 ** 53)

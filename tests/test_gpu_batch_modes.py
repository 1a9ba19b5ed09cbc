"""The two ways a batch steps, one launch per step and the persistent kernel: which one
runs, the way from one to the other, and the same fields as lattices stepped alone."""
import ctypes
import json

import pytest

from paper_2402_15752_gb300 import Batch, Simulation
from paper_2402_15752_gb300 import workloads as wl

from test_gpu_batch import _assert_same, _cases, _sims

pytestmark = pytest.mark.gpu


def _squares(sides, **over):
    return [wl.droplet64(nx=n, ny=n, R=0.3 * n, **over) for n in sides]


@pytest.mark.parametrize("sides,per_step", [([64] * 4, True), ([768] * 8, False)])
def test_the_batch_says_how_it_steps(sides, per_step):
    # 8 x 768^2: 2304 tiles of 128 x 16, two for each of 7 CTAs per SM, no idle column
    cases = _squares(sides)
    sims, alone = _sims(cases), _sims(cases)
    b = Batch(sims)
    t = b.tiling()
    assert t["per_step"] is per_step
    assert (t["tile_w"], t["tile_h"]) == (128, 16)
    b.step(5)
    b.sync()
    for s in alone:
        s.step(5)
    _assert_same(sims, alone, label="default mode")
    b.set_tiling(64, 16)
    assert not b.tiling()["per_step"]
    b.close()
    assert b.L.lbm_batch_per_step(ctypes.c_void_p()) == -1


def test_default_waits_leave_the_launches_per_step():
    cases = _cases()
    sims, alone = _sims(cases), _sims(cases)
    b = Batch(sims)
    assert b.tiling()["per_step"]
    b.step(3)
    b.set_wait_limit(1 << 21, -1)  # the defaults
    assert b.tiling()["per_step"]
    b.step(4)
    b.set_wait_limit(1 << 20, -1)  # 7 steps in: a limit, and back after an odd number of steps
    assert not b.tiling()["per_step"]
    b.step(35)
    b.set_wait_limit(1 << 21, -1)
    assert b.tiling()["per_step"]
    b.step(33)
    b.set_tiling(32, 8)  # the persistent kernel by choice: the defaults leave it
    b.set_wait_limit(1 << 21, -1)
    assert not b.tiling()["per_step"]
    b.step(6)
    b.sync()
    for s in alone:
        s.step(3 + 4 + 35 + 33 + 6)
    _assert_same(sims, alone, label="modes in turn")
    b.close()


def _us(b, n=32):
    """us per step, the best of 6 runs of n steps."""
    import torch
    best = float("inf")
    for _ in range(6):
        a, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        b.step(n)
        e.record()
        e.synchronize()
        best = min(best, a.elapsed_time(e) * 1e3 / n)
    return best


@pytest.mark.parametrize("q", [5, 9])
def test_a_tuned_batch_is_not_slower_than_it_was(q, tmp_path):
    # 4 x 64^2: some 3 us a step by launches, some 10 in the best persistent tiling
    cases = _squares([64] * 4, scalar_q=q)
    sims, alone = _sims(cases), _sims(cases)
    b = Batch(sims)
    before = _us(b)
    cache = str(tmp_path / "tiles.json")
    got = b.autotune(steps_per_trial=4, cache=cache)
    assert got["per_step"] and b.tiling()["per_step"]
    assert len(got["trials"]) == 12 and all(s.time == 192 + 12 * 6 for s in sims)
    assert _us(b) < 2 * before
    for s in alone:
        s.step(sims[0].time)
    _assert_same(sims, alone, label="after autotune")
    # from the cache, on a batch that was moved away, and from a cache without the mode
    b.set_tiling(32, 4)
    again = b.autotune(cache=cache)
    assert again["cached"] and again["per_step"] and b.tiling()["per_step"]
    known = json.load(open(cache))
    json.dump({b.signature(): known[b.signature()]}, open(cache, "w"))
    assert b.autotune(cache=cache)["per_step"]
    b.set_per_step(False)
    assert not b.autotune(cache=cache)["per_step"]
    b.close()


def test_a_tuned_batch_with_limited_waits_keeps_the_persistent_kernel():
    cases = _cases()[:3]
    sims, alone = _sims(cases), _sims(cases)
    b = Batch(sims)
    b.set_wait_limit(1 << 20, -1)
    got = b.autotune(steps_per_trial=3)
    assert not got["per_step"] and all(s.time == 60 for s in sims)
    b.set_per_step(True)  # takes effect with the default waits
    assert not b.tiling()["per_step"]
    b.step(3)
    b.set_wait_limit(1 << 21, -1)
    assert b.tiling()["per_step"]
    b.step(3)
    b.sync()
    for s in alone:
        s.step(66)
    _assert_same(sims, alone, label="limited, then not")
    b.close()


@pytest.mark.parametrize("q", [5, 9])
def test_ragged_walled_lattices_by_launches(q):
    cases = [wl.droplet64(nx=nx, ny=ny, R=0.3 * min(nx, ny), scalar_q=q, wall_x=wx, wall_y=wy, rho2=0.5, Fx=1e-6)
             for nx, ny, wx, wy in ((33, 31, 1, 1), (64, 5, 0, 1), (7, 130, 1, 0), (100, 61, 0, 0), (1, 9, 0, 1), (65, 1, 1, 0))]
    sims, alone = _sims(cases), _sims(cases)
    b = Batch(sims)
    assert b.tiling()["per_step"]
    b.step(7)
    b.step(70)  # two graphs of 32 steps from an odd step, six launches
    b.sync()
    for s in alone:
        s.step(77)
    _assert_same(sims, alone, label="launches per step, D2Q%d" % q)
    b.close()

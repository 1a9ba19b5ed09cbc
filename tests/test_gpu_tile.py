"""The tile step kernels at the edges of their tiles and at the lines between the step
kernels: odd and one-node-wide lattices against the oracle, and a periodic lattice
against itself repeated until another kernel (or tile) steps it."""
import numpy as np
import pytest

import oracle
from paper_2402_15752_gb300 import Simulation
from paper_2402_15752_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "fp32": 1e-5}


def _case(nx, ny, **over):
    w = wl.droplet64(nx=nx, ny=ny, R=0.3 * min(nx, ny) + 1, **over)
    g = np.random.default_rng(nx * 1000 + ny)
    phi = 0.5 + 0.5 * np.tanh(w.sdf / 2)
    u = [1e-2 * np.sin(2 * np.pi * (np.arange(nx) / nx))[None, :] + np.zeros((ny, nx)),
         1e-2 * np.cos(2 * np.pi * (np.arange(ny) / ny))[:, None] + np.zeros((ny, nx))]
    p = 1e-4 * g.standard_normal((ny, nx))
    return w, [np.ascontiguousarray(a) for a in (phi, u[0], u[1], p, phi, 0.3 * (1 - phi))]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("q", [5, 9])
@pytest.mark.parametrize("nx,ny,wx,wy", [(1, 1, 0, 0), (2, 3, 1, 0), (7, 4, 0, 1), (8, 5, 1, 1), (17, 9, 0, 0),
                                         (31, 4, 1, 0), (33, 7, 0, 1), (97, 61, 1, 1), (1, 50, 0, 1), (70, 1, 1, 0)])
def test_tiles_against_the_oracle(nx, ny, wx, wy, q, precision):
    # visc_model cycles through the three relations with the size
    over = dict(wall_x=wx, wall_y=wy, scalar_q=q, visc_model=(nx + ny) % 3, visc_beta=0.5, rho1=1.0, rho2=0.2, mu1=0.2,
                mu2=0.1, Fx=1e-6, gy=-1e-6)
    w, m = _case(nx, ny, **over)
    ref = oracle.OracleSim(w.params)
    ref.init_macros(*m)
    ref.step(7)
    want = ref.fields()
    sim = Simulation(w.params, precision=precision)
    sim.init_macros(*m)
    sim.step(7)
    got = sim.fields()
    sim.sync()
    # natural scales, as in the parity tests
    speed, pmax = np.hypot(want["ux"], want["uy"]).max(), np.abs(want["p"]).max()
    us, total = max(speed, pmax * 3 ** 0.5), np.abs(want["c1"] + want["c2"]).max()
    scale = dict(phi=1.0, ux=us, uy=us, p=max(pmax, speed / 3 ** 0.5), c1=total, c2=total, rho=1.0,
                 mu=np.abs(want["mu"]).max())
    for k, s in scale.items():
        assert np.abs(got[k] - want[k]).max() <= TOL[precision] * s, k
    sim.close()


# (precision, side, repeats): FP32 D2Q5 tiles against strips (700 000 nodes), FP64 tiles of
# 8 x 4 against 16 x 8 (two per SM)
@pytest.mark.parametrize("precision,side,times", [("fp32", 160, 6), ("fp64", 64, 4)])
def test_a_repeated_lattice_steps_alike(precision, side, times):
    w, m = _case(side, side, Fx=1e-6)
    out = []
    for n in (1, times):
        sim = Simulation(dict(w.params, nx=n * side, ny=n * side), precision=precision)
        sim.init_macros(*[np.ascontiguousarray(np.tile(a, (n, n))) for a in m])
        sim.step(9)
        out.append(sim.fields())
        sim.close()
    for k, a in out[0].items():
        np.testing.assert_array_equal(out[1][k], np.tile(a, (times, times)), err_msg=k)


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16", "fp16"])
def test_a_non_finite_state_is_reported(precision):
    from paper_2402_15752_gb300.lbm import LBMError
    w, m = _case(40, 24)
    m[1][5, 7] = np.nan
    sim = Simulation(w.params, precision=precision)
    sim.init_macros(*m)
    sim.step(1)
    with pytest.raises(LBMError) as e:
        sim.sync()
    assert e.value.code == -5
    sim.close()

"""A NaN of the state shows in every field that it enters, in each storage precision
whose kernels evaluate the fields, whatever its sign."""
import numpy as np
import pytest

from paper_2402_15752_gb300 import Simulation
from paper_2402_15752_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("visc_model", [0, 1, 2])
@pytest.mark.parametrize("q", [5, 9])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny", [(24, 16), (200, 120)])
def test_a_nan_scalar_or_flow_shows_in_the_fields(nx, ny, precision, q, visc_model, sign):
    w = wl.droplet64(nx=nx, ny=ny, R=5.0, scalar_q=q, visc_model=visc_model, visc_beta=0.5, rho2=0.5, mu2=0.05)
    phi = np.ascontiguousarray(0.5 + 0.5 * np.tanh(w.sdf / 2))
    z = np.zeros_like(phi)
    y0, x0 = ny // 2, nx // 2
    bad = np.copysign(np.nan, sign)

    def at(fields):
        sim = Simulation(w.params, precision=precision)
        sim.init_macros(*[np.ascontiguousarray(a) for a in fields])
        f = sim.fields()
        sim.close()
        return {k: v[y0, x0] for k, v in f.items()}
    c1 = phi.copy()
    c1[y0, x0] = bad
    got = at((phi, z, z, z, c1, 0.3 * (1 - phi)))
    assert np.isnan(got["c1"]) and np.isnan(got["c2"])
    assert np.isnan(got["mu"]) == (visc_model != 0) and np.isfinite(got["rho"])
    ux = z.copy()
    ux[y0, x0] = bad
    got = at((phi, ux, z, z, phi, 0.3 * (1 - phi)))
    # FP64 stores phi as a double, and a NaN velocity reaches f: the node's phi is NaN.  The
    # fixed point of FP32 holds no NaN.
    names = ("phi", "ux", "uy", "p", "c1", "c2", "rho") if precision == "fp64" else ("ux", "uy", "p", "c1", "c2")
    for k in names:
        assert np.isnan(got[k]), k
    if precision == "fp64" and visc_model == 0:
        assert np.isnan(got["mu"])


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("q", [5, 9])
def test_a_nan_phase_field_shows_in_the_fields(q, sign):
    w = wl.droplet64(nx=24, ny=16, R=5.0, scalar_q=q, rho2=0.5, mu2=0.05)
    phi = np.ascontiguousarray(0.5 + 0.5 * np.tanh(w.sdf / 2))
    phi[8, 12] = np.copysign(np.nan, sign)
    sim = Simulation(w.params, precision="fp64")
    sim.init_fields(phi, np.ones_like(phi), np.ones_like(phi))
    got = sim.fields()
    for k in ("phi", "ux", "uy", "p", "c1", "c2", "rho", "mu"):
        assert np.isnan(got[k][8, 12]), k
    sim.close()

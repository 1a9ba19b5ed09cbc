"""The strip kernels on the lattices that still step in strips: FP64 and D2Q9 scalars
only where the tiles' offsets or their grid end (2^31 words of populations, 262 140
rows), FP32 and 16-bit D2Q5 on large lattices.  Against the oracle, in the release and
the bounds-checked build.

A lattice 4 nodes wide and 262 144 rows tall is 64 rows repeated: it steps like the
4 x 64 lattice, which the oracle runs.  Tolerances, relative to each field's natural scale:
the parity bars in FP64 and FP32; in 16-bit storage, where the rounding depends on the
node, the bars by which two builds of those kernels may differ.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_2402_15752_gb300 import Batch, Simulation
from paper_2402_15752_gb300 import workloads as wl

from _parity import MAIN_FIELDS, field_scales, rel_max_errors
from test_gpu_tile import _case

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "fp32": 1e-5, "fp16": 5e-3, "bf16": 5e-2}
TALL = [("fp64", 5, 0), ("fp64", 5, 1), ("fp64", 9, 0), ("fp64", 9, 1), ("fp32", 9, 0), ("fp32", 9, 1), ("bf16", 5, 0),
        ("bf16", 9, 1), ("fp16", 9, 0)]
STEPS = 7
OVER = dict(rho1=1.0, rho2=0.2, mu1=0.2, mu2=0.1, Fx=1e-6, gy=-1e-6)


def _oracle(w, m, steps):
    ref = oracle.OracleSim(w.params)
    ref.init_macros(*m)
    ref.step(steps)
    return ref.fields()


def _run(w, m, precision, ny):
    """Fields and conserved sums of the lattice m repeated to ny rows."""
    times = ny // m[0].shape[0]
    sim = Simulation(dict(w.params, ny=ny), precision=precision)
    sim.init_macros(*[np.ascontiguousarray(np.tile(a, (times, 1))) for a in m])
    sim.step(STEPS)
    sim.sync()
    f = sim.fields()
    sim.close()
    return f


@pytest.mark.parametrize("precision,q,wall_x", TALL)
def test_a_tall_lattice_against_the_oracle(precision, q, wall_x):
    w, m = _case(4, 64, scalar_q=q, wall_x=wall_x, **OVER)
    want = _oracle(w, m, STEPS)
    got = _run(w, m, precision, 262144)
    names = MAIN_FIELDS + ("rho", "mu")
    errs = rel_max_errors({k: got[k].reshape(4096, 64, 4) for k in names}, want, names)
    assert max(errs.values()) <= TOL[precision], errs


@pytest.mark.parametrize("wx,wy", [(1, 1), (0, 1), (1, 0)])
def test_a_wide_odd_lattice_with_walls_against_the_oracle(wx, wy):
    # 703 703 nodes; the last strip has 105 of its 128 columns
    w, m = _case(1001, 703, wall_x=wx, wall_y=wy, **OVER)
    got = _run(w, m, "fp32", 703)
    errs = rel_max_errors(got, _oracle(w, m, STEPS), MAIN_FIELDS + ("rho", "mu"))
    assert max(errs.values()) <= TOL["fp32"], errs


# 8192 columns: the last rows of the tiles' 32-bit offsets and the first lattices beyond
@pytest.mark.parametrize("precision,q,ny", [("fp32", 9, 7280), ("fp32", 9, 7300), ("fp64", 5, 9360), ("fp64", 5, 9380)])
def test_both_sides_of_the_offsets_end(precision, q, ny):
    import torch
    w, m = _case(64, 20, scalar_q=q, **OVER)
    steps = 3
    want = _oracle(w, m, steps)
    sim = Simulation(dict(w.params, nx=8192, ny=ny), precision=precision)
    values = (8192 // 32) * ny * 32 * (18 + 2 * q)
    assert (values >= 1 << 31) == (ny in (7300, 9380))
    sim.init_macros(*[torch.from_numpy(a).cuda().repeat(ny // 20, 128) for a in m])
    b = Batch([sim]) if precision == "fp32" else None
    if b and values >= 1 << 31:  # the batch's launches take the same offsets
        assert not b.tiling()["per_step"]
    (b or sim).step(1)
    sim.step(steps - 1)
    sim.sync()
    scale = field_scales(want)
    for k in MAIN_FIELDS + ("rho", "mu"):
        f = sim.fields(names=(k,), device=True)[k].view(ny // 20, 20, 128, 64)
        d = (f - torch.from_numpy(want[k]).cuda()[None, :, None, :]).abs().max().item()
        assert d <= TOL[precision] * scale[k], (k, d)
    if b:
        b.close()
    sim.close()


CHILD = """
import sys
import numpy as np
sys.path[:0] = [%r, %r]
import test_gpu_strips as t
out = {}
for precision, q, wall_x in t.TALL:
    w, m = t._case(4, 64, scalar_q=q, wall_x=wall_x, **t.OVER)
    f = t._run(w, m, precision, 262144)  # sync raises on an access outside the workspace
    for k in t.MAIN_FIELDS:
        out["%%s_%%d_%%d_%%s" %% (precision, q, wall_x, k)] = f[k][:512]
w, m = t._case(1001, 703, wall_x=1, wall_y=1, **t.OVER)
f = t._run(w, m, "fp32", 703)
for k in t.MAIN_FIELDS:
    out["wide_" + k] = f[k]
from paper_2402_15752_gb300 import lbm
out["debug"] = np.array(int(lbm.load_library().lbm_debug_build()))
np.savez(sys.argv[1], **out)
"""


def test_the_strips_stay_inside_the_workspace(tmp_path):
    from paper_2402_15752_gb300 import build
    build.build()
    build.build(debug=True)
    here = os.path.dirname(os.path.abspath(__file__))
    runs = []
    for debug in "01":
        out = str(tmp_path / ("run%s.npz" % debug))
        r = subprocess.run([sys.executable, "-c", CHILD % (here, os.path.dirname(here)), out],
                           env=dict(os.environ, LBM_DEBUG=debug), capture_output=True, text=True, timeout=900)
        assert r.returncode == 0, (r.stdout[-3000:], r.stderr[-3000:])
        runs.append(dict(np.load(out)))
    assert [int(r["debug"]) for r in runs] == [0, 1]
    keys = ["%s_%d_%d" % c for c in TALL]
    for key, precision in [(k, k.split("_")[0]) for k in keys] + [("wide", "fp32")]:
        errs = rel_max_errors(*[{k: r[key + "_" + k] for k in MAIN_FIELDS} | {"rho": np.ones(1)} for r in runs], MAIN_FIELDS)
        assert max(errs.values()) <= TOL[precision], (key, errs)

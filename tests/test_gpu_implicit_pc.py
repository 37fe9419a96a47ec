"""Windowed FP32 preconditioner, linearised Jacobian products and fused
Gram-Schmidt passes of the backward-Euler solve at sizes around their windows
(32 x 32 less two halos of 1 to 8 cells), blocks and restarts.

The FP64 preconditioner (pc_precision "fp64") runs one kernel per step and
shares no code with the windowed one.  Both solves end at the same Newton
rule (max |F| <= 1e-12), so the fields agree to 1e-9, the bound that the
comparison with the oracle uses at these parameters.  The iteration counts
are compared at the mild time step only (10 % and 3 per Newton step): at
dt D ~ 3e4 the two preconditioners differ by FP32 rounding times the blocks'
conditioning, and the last systems' right-hand sides are at rounding level."""
import numpy as np
import pytest

from paper_2111_11538_gb300 import Simulation, inputs, native, workloads

pytestmark = pytest.mark.gpu

KEYS = ("theta", "xO", "xH", "xW")


@pytest.fixture(scope="module", autouse=True)
def _built():
    native.build_library()
    native.lib()


def _run(shape, dt, **kw):
    f = inputs.core_shell(shape, 0.3 * min(shape), 0.1 * min(shape) + 0.5, delta=1.5)
    sim = Simulation(shape, workloads.paper_params(cg_rtol=1e-12), precision="fp64")
    sim.set_fields(f)
    st = sim.step_implicit(1, dt, **kw)
    g = sim.get_fields(keys=KEYS)
    sim.close()
    return g, st


@pytest.mark.parametrize("shape,degree,restart", [
    ((7, 5), 32, 60), ((24, 24), 32, 60), ((25, 47), 32, 60), ((33, 70), 31, 60), ((64, 31), 9, 60),
    ((40, 16), 32, 7), ((18, 90), 64, 60), ((30, 30), 1, 60), ((6, 9, 7), 32, 60)])
def test_windowed_preconditioner_matches_fp64(shape, degree, restart):
    dt = 0.05 if degree > 16 else 1e-4
    kw = dict(pc_degree=degree, gmres_restart=restart)
    g, s = _run(shape, dt, pc_precision="mixed", **kw)
    r, t = _run(shape, dt, pc_precision="fp64", **kw)
    for k in KEYS:
        assert np.linalg.norm(g[k] - r[k]) <= 1e-9 * np.linalg.norm(r[k]), k
    assert abs(s["newton_iters"] - t["newton_iters"]) <= 1
    if dt < 1e-3:
        assert abs(s["gmres_iters"] - t["gmres_iters"]) <= 0.1 * t["gmres_iters"] + 3 * t["newton_iters"], (s, t)

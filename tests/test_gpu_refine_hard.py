"""Mixed solves with the Jacobi preconditioner on 2D grids whose condition
number leaves an FP32 pass little: every pass's target has to be one that it can
reach, or it runs on to cg_maxit.  rtol 1e-10, from rest and with the
extrapolated guess; core-shells of several radii, shell thicknesses and
positions."""
import numpy as np
import pytest

from paper_2111_11538_gb300 import Simulation, inputs, native, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    native.build_library()
    native.lib()


@pytest.mark.parametrize("shape", [(138, 224), (241, 255), (206, 414)])
def test_jacobi_passes_reach_their_targets(shape):
    rng = np.random.default_rng(5)
    prm = workloads.params(plasticity=1, cg_rtol=1e-10, warm_start="extrap", precond="jacobi")
    sim = Simulation(shape, prm, precision="mixed")
    for k in range(6):
        n = min(shape)
        f = inputs.core_shell(shape, n * rng.uniform(0.28, 0.34), n * rng.uniform(0.05, 0.08))
        cut = tuple(rng.integers(0, s) for s in shape)
        f = {key: np.ascontiguousarray(np.roll(v, cut, (0, 1))) for key, v in f.items()}
        sim.set_fields(f)
        sim.step(3)
        assert sim.diagnostics()["cg_rel_residual"] <= 1e-10, k
    sim.close()

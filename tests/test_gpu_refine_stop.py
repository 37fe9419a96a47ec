"""Where the mixed method's refinement stops: PF_OK means that the returned
solution's FP64 residual has met cg_rtol, also if cg_maxit ends the pass that
follows the one that met it, and at tolerances where rounding can take a
residual that was met above the tolerance again."""
import numpy as np
import pytest

from paper_2111_11538_gb300 import Simulation, inputs, native, workloads

pytestmark = pytest.mark.gpu

CASES = [((24, 20), "jacobi"), ((32, 48), "mg"), ((10, 9, 8), "jacobi"), ((16, 16, 32), "mg")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    native.build_library()
    native.lib()


def _solve(shape, precond, rtol, maxit):
    f = inputs.core_shell(shape, 0.3 * min(shape), 0.1 * min(shape) + 1.0, delta=1.5)
    sim = Simulation(shape, workloads.params(cg_rtol=rtol, cg_maxit=maxit, prestress=0.01, precond=precond),
                     precision="mixed")
    sim.set_fields(f)
    rc = sim.step(1, check=False)
    d = sim.diagnostics() if rc == native.PF_OK else None
    sim.close()
    assert rc in (native.PF_OK, native.PF_ENOTCONV)
    return d


@pytest.mark.parametrize("shape,precond", CASES)
def test_capped_solve_meets_its_tolerance(shape, precond):
    for rtol in np.geomspace(3e-7, 1e-9, 16):
        d = _solve(shape, precond, rtol, 20000)
        assert d["cg_rel_residual"] <= rtol
        n = d["cg_iters_last"]
        for maxit in range(max(1, n - 12), n):
            c = _solve(shape, precond, rtol, maxit)
            assert c is None or c["cg_rel_residual"] <= rtol, (rtol, maxit, c["cg_rel_residual"])


@pytest.mark.parametrize("shape,precond", CASES)
def test_tolerance_near_the_rounding_of_the_residual(shape, precond):
    met = 0
    for rtol in np.geomspace(1e-13, 2e-16, 60):
        d = _solve(shape, precond, rtol, 4000)
        assert d is None or d["cg_rel_residual"] <= rtol, (rtol, d["cg_rel_residual"])
        met += d is not None
    assert met > 0

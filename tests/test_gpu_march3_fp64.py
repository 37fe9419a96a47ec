"""3D mixed solves (warp-marching FP32 sweeps) against the FP64 Jacobi solve,
whose operator comes from the element matrices and shares no code with them:
x sizes below, at and past a strip's 30 columns and a periodic strip's 32, odd
rows and planes, the smallest grids.

The mixed solve's residual is measured in FP64, so a wrong sweep shows in its
iterations: a solve of rtol 1e-8 takes at most four FP32 passes, none longer
than the FP64 solve's to 1e-10.  Fields: FP32 storage, 1e-5; sigma, linear in u
(cond * rtol of it, cond <= 1e4 here), 1e-3 of its size."""
import numpy as np
import pytest

from paper_2111_11538_gb300 import Simulation, inputs, native, workloads

pytestmark = pytest.mark.gpu

KEYS = ["phi_f", "phi_w", "xO", "xH", "xW"]
JACOBI = [(2, 2, 2), (3, 2, 5), (5, 4, 29), (4, 7, 30), (6, 5, 31), (3, 4, 32), (7, 3, 33), (2, 9, 60), (5, 6, 61),
          (4, 5, 64), (9, 11, 93)]
MG = [(8, 8, 34), (16, 16, 60), (16, 34, 62), (18, 16, 64), (16, 16, 92)]


def rel(a, b):
    a, b = np.asarray(a, float), np.asarray(b, float)
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


@pytest.fixture(scope="module", autouse=True)
def _built():
    native.build_library()
    native.lib()


def _run(shape, precision, precond, rtol):
    f = inputs.core_shell(shape, 0.35 * min(shape), 0.1 * min(shape) + 0.7, delta=1.5)
    prm = workloads.params(plasticity=1, sigma_Y=0.004, H_hard=0.01, cg_rtol=rtol, prestress=0.01, precond=precond)
    sim = Simulation(shape, prm, precision=precision)
    sim.set_fields(f)
    sim.step(2)
    g, d = sim.get_fields(), sim.diagnostics()
    sim.close()
    return g, d


@pytest.mark.parametrize("shape,precond", [(s, "jacobi") for s in JACOBI] + [(s, "mg") for s in MG])
def test_mixed_matches_fp64_element_matrices(shape, precond):
    ref, dr = _run(shape, "fp64", "jacobi", 1e-10)
    g, d = _run(shape, "mixed", precond, 1e-8)
    for k in KEYS:
        assert rel(g[k], ref[k]) < 1e-5, (k, rel(g[k], ref[k]))
    assert rel(g["sigma"], ref["sigma"]) < 1e-3
    assert d["cg_iters_max"] <= 4 * dr["cg_iters_max"] + 8, (d["cg_iters_max"], dr["cg_iters_max"])

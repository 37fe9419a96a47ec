"""Warp-marching V-cycle sweeps at the sizes where their strips, rows, chunks
and halos can go wrong: a grid narrower than a warp (periodic strip), one
column short of, at and past a strip's 28 or 30 columns, odd rows and planes,
one level, and coarse levels with odd sizes.  The multigrid solve has to meet
the same systems as the Jacobi solve, whose kernel shares none of this code.

Tolerances: both solves end at ||r|| <= rtol ||b|| (the mixed method measures
its residual in FP64 and stores the displacement in FP32); the error of u is
at most cond * rtol of it, cond <= 1e4 at these sizes, which the fields see
through the mechanical driving force scaled by dt * M ~ 1e-2.  fp64, rtol 1e-10:
1e-8.  mixed, rtol 1e-8: fields to the 1e-5 that FP32 storage already costs.
The stress, linear in u, gets the factor 1e3 (1e-5, 1e-2 of its largest value)."""
import numpy as np
import pytest

from paper_2111_11538_gb300 import Batch, Simulation, inputs, native, workloads

pytestmark = pytest.mark.gpu

KEYS = ["phi_f", "phi_w", "xO", "xH", "xW"]
SHAPES = [
    (16, 34), (28, 20), (30, 38), (32, 30), (34, 26),      # periodic strip up to 32, two strips from 33
    (56, 22), (58, 44), (60, 36), (62, 90),                # 28- and 30-column strips, remainders of 2
    (31, 37), (90, 118),                                   # one level; odd sizes below the finest
    (32, 32, 8), (30, 12, 10), (34, 10, 14),               # 3D: strips of 30
    (62, 6, 18), (28, 22, 6), (35, 9, 7),
]


def rel(a, b):
    a, b = np.asarray(a, float), np.asarray(b, float)
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


@pytest.fixture(scope="module", autouse=True)
def lib():
    native.build_library()
    native.lib()


def _run(shape, prm, f, precision, precond):
    sim = Simulation(shape, dict(prm, precond=precond), precision=precision)
    sim.set_fields(f)
    sim.step(3)
    g, d = sim.get_fields(), sim.diagnostics()
    sim.close()
    return g, d


@pytest.mark.parametrize("precision,rtol,tol", [("fp64", 1e-10, 1e-8), ("mixed", 1e-8, 1e-5)])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_sweeps_match_jacobi(shape, precision, rtol, tol):
    f = inputs.core_shell(shape, 0.3 * min(shape), 0.1 * min(shape) + 1.0, delta=1.5)
    prm = workloads.params(plasticity=1, sigma_Y=0.004, H_hard=0.01, cg_rtol=rtol, prestress=0.01)
    gj, _ = _run(shape, prm, f, precision, "jacobi")
    gm, d = _run(shape, prm, f, precision, "mg")
    assert d["precond"] == native.PF_PC_MG
    for k in KEYS:
        assert rel(gm[k], gj[k]) < tol, (k, rel(gm[k], gj[k]))
    assert rel(gm["sigma"], gj["sigma"]) < 1e3 * tol, rel(gm["sigma"], gj["sigma"])
    assert rel(gm["Ebar"], gj["Ebar"]) < 1e3 * tol


def test_large_3d_batch_in_two_launches():
    """A batch of more 3D mixed instances than the device has SMs (their CG
    blocks take an SM each) runs in two launches; every instance ends where a
    solve of its own does.  The two differ in the blocks that share the work
    and so in the rounding of FP32 sums: 1e-5, as for the solves above."""
    shapes = [(8, 8, 8), (16, 8, 10)] * 100
    prm = workloads.params(plasticity=1, sigma_Y=0.004, H_hard=0.01, cg_rtol=1e-8, precond="mg")
    fields = {s: inputs.core_shell(s, 2.4, 1.8, delta=1.5) for s in set(shapes)}
    b = Batch(shapes, prm, precision="mixed")
    for i, s in enumerate(shapes):
        b.set_fields(i, fields[s])
    b.step(2)
    ref = {}
    for s in set(shapes):
        sim = Simulation(s, prm, precision="mixed")
        sim.set_fields(fields[s])
        sim.step(2)
        ref[s] = sim.get_fields()
        sim.close()
    for i in (0, 1, 98, 99, 100, 101, 198, 199):
        got = b.get_fields(i)
        for k in KEYS:
            assert rel(got[k], ref[shapes[i]][k]) < 1e-5, (i, k)
        assert rel(got["sigma"], ref[shapes[i]]["sigma"]) < 1e-2
    b.close()

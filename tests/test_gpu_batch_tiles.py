"""2D batches of more Jacobi-preconditioned mixed instances than SMs, whose first
grid alone would take a CG block of 512 threads, one to an SM; every instance
ends where a solve of its own does (1e-5: FP32 storage)."""
import numpy as np
import pytest

from paper_2111_11538_gb300 import Batch, Simulation, inputs, native, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    native.build_library()
    native.lib()


def test_batch_of_more_instances_than_sms():
    shapes = [(137, 321)] + [(9, 7), (13, 18)] * 110
    prm = workloads.params(cg_rtol=1e-8, prestress=0.01, precond="jacobi")
    fields = {s: inputs.core_shell(s, 0.3 * min(s), 0.1 * min(s) + 0.5, delta=1.5) for s in set(shapes)}
    b = Batch(shapes, prm, precision="mixed")
    for i, s in enumerate(shapes):
        b.set_fields(i, fields[s])
    b.step(1)
    for i in (0, 1, 2, 219, 220):
        sim = Simulation(shapes[i], prm, precision="mixed")
        sim.set_fields(fields[shapes[i]])
        sim.step(1)
        ref, got = sim.get_fields(), b.get_fields(i)
        sim.close()
        for k in ("phi_f", "xO", "xH"):
            assert np.linalg.norm(got[k] - ref[k]) <= 1e-5 * np.linalg.norm(ref[k]), (i, k)
    b.close()

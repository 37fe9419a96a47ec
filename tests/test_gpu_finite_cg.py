"""The finite-strain CG kernel over several rounds of cells per block.

A periodic problem repeated m times along each axis has the repeated solution
(the equilibrium with u = 0 at node 0 is unique), so a large grid is checked
against a small one that needs one round of a few blocks, which the oracle
covers.  The mean-deformation rows of the residual are sums over all cells, so
the large solve's max |residual| cannot go below N 1e-16 times the stresses; it
ends at 1e-11, the small one at 1e-13.  The smallest eigenvalue of the elastic
operator on a grid of 210 nodes is above 1e-4, so u agrees to 1e-7, |u| being
~0.1: 1e-6 of the largest u.  Fbar, whose rows carry a factor N: 1e-10."""
import numpy as np
import pytest

from paper_2111_11538_gb300 import make_config, native, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    native.build_library()
    native.lib()


def _solve(th, pg, precision, tol):
    o = native.pf_fs_opts(nload=2, newton_maxit=40, newton_tol=tol, cg_maxit=20000, cg_rtol=1e-12,
                          precision=precision)
    rc, u, Fb, st = native.pf_finite_strain_solve(make_config(th.shape, workloads.params(prestress=0.003)), th.ravel(),
                                                  pg.ravel(), 0.2, None, o)
    assert rc == native.PF_OK, native.lib().pf_fs_last_error()
    return np.asarray(u).reshape(th.shape + (th.ndim,)), Fb


@pytest.mark.parametrize("shape,reps", [((3, 2, 4), (15, 16, 10)), ((5, 4, 3), (9, 10, 8)), ((7, 6), (30, 31)),
                                        ((2, 2), (1, 1)), ((2, 3, 2), (1, 2, 1))])
@pytest.mark.parametrize("precision", [native.PF_MIXED, native.PF_FP64])
def test_repeated_problem(shape, reps, precision):
    rng = np.random.default_rng(sum(shape))
    th = np.clip(0.5 + 0.4 * rng.standard_normal(shape), 0.0, 1.0)
    pg = np.zeros(shape)
    pg.flat[1] = 0.7
    th.flat[1] = 0.0
    u0, F0 = _solve(th, pg, native.PF_FP64, 1e-13)
    u, F = _solve(np.tile(th, reps), np.tile(pg, reps), precision, 1e-11)
    scale = np.abs(u0).max()
    assert np.abs(u - np.tile(u0, reps + (1,))).max() <= 1e-6 * scale
    assert np.abs(F - F0).max() <= 1e-10

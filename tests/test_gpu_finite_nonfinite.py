"""A finite-strain residual that is not finite is not an equilibrium, whether
one cell or every cell makes it so."""
import numpy as np
import pytest

from paper_2111_11538_gb300 import make_config, native, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    native.build_library()
    native.lib()


@pytest.mark.parametrize("shape", [(6, 5), (4, 5, 6)])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("cells", [1, None])
@pytest.mark.parametrize("precision", [native.PF_MIXED, native.PF_FP64])
def test_nonfinite_residual_is_not_converged(shape, bad, cells, precision):
    th, pg = np.full(shape, 0.5), np.zeros(shape)
    th.flat[:cells] = bad
    o = native.pf_fs_opts(nload=1, newton_maxit=3, newton_tol=1e-10, cg_maxit=50, cg_rtol=1e-8, precision=precision)
    rc, u, Fb, st = native.pf_finite_strain_solve(make_config(shape, workloads.params(prestress=0.003)), th.ravel(),
                                                  pg.ravel(), 0.2, None, o)
    assert rc == native.PF_ENOTCONV
    assert not np.isfinite(st.residual)

"""Grid sizes that the library's index arithmetic covers: a vector's 3 N values
in 32 bits in the 3D mixed solve, 2^31 cells elsewhere (checked before any
device call)."""
import pytest
import torch

from paper_2111_11538_gb300 import make_config, native, workloads


@pytest.fixture(scope="module", autouse=True)
def _lib():
    native.build_library()
    native.lib()


def _create(shape, precision, mechanics):
    rc, h = native.pf_create(make_config(shape, workloads.params(mechanics=mechanics), precision=precision))
    assert not h.value
    return rc, native.pf_last_error(None)


def test_3d_mixed_mechanics_limit():
    rc, err = _create((700, 1024, 2048), "mixed", 1)
    assert rc == native.PF_EINVAL and "2^32" in err


@pytest.mark.skipif(torch.cuda.is_available(), reason="would allocate the grid")
@pytest.mark.parametrize("shape,precision,mechanics", [
    ((1365, 1024, 1024), "mixed", 1), ((700, 1024, 2048), "mixed", 0), ((700, 1024, 2048), "fp64", 1),
    ((32768, 65536), "mixed", 1)])
def test_other_grids_pass_the_size_check(shape, precision, mechanics):
    assert _create(shape, precision, mechanics)[0] == native.PF_ECUDA

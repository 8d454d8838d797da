"""Which kernel a handle takes: small lattices the direct one whatever their options, and
lattices with small planes the faster of the two whatever their size."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("strain_mode", [0, 1])
def test_small_lattices(gpu_lib, precision, strain_mode):
    p = gpu_lib.make_params(16, nu0=0.01, cs=0.13, precision=precision, strain_mode=strain_mode)
    with gpu_lib.Lattice(p) as L:
        assert L.config()["kind"] == 1

"""lbm_kernel_config of a direct-kernel handle: it has no tiles, so it reports the rows that
were asked for, or none."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [0, 1, 3])
def test_tile_rows_of_the_direct_kernel(gpu_lib, rows):
    with gpu_lib.Lattice(gpu_lib.make_params(12, nu0=0.01, kernel=1, tile_rows=rows, threads=128)) as L:
        assert L.config()["tile_rows"] == rows
        L.init(gpu_lib.LBM_INIT_TGV3D, amplitude=0.02)
        L.step(2)
        assert L.theta_slice(2, 11).shape == (12, 12)

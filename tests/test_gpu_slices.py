"""Slices on both sides of the size from which they are widened on the device."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(4, 257, 255), (4, 256, 256), (3, 90, 800), (70, 4, 1000)])  # nz, ny, nx
@pytest.mark.parametrize("cfg", [dict(kernel=1, tile_rows=1, threads=128), dict(kernel=2, tile_rows=1, stages=2, threads=256)])
def test_slices_are_planes_of_the_field(gpu_lib, shape, cfg):
    nz, ny, nx = shape
    rng = np.random.default_rng(1)
    with gpu_lib.Lattice(gpu_lib.make_params(nx, ny, nz, nu0=0.01, cs=0.13, **cfg)) as L:
        L.init(gpu_lib.LBM_INIT_VELOCITY, u=rng.normal(scale=0.02, size=(3, *shape)))
        L.step(3)
        theta = L.fields()["theta"]
        for axis, n in ((0, nx), (1, ny), (2, nz)):
            for k in (0, n - 1):
                assert np.array_equal(L.theta_slice(axis, k), np.take(theta, k, axis=2 - axis))

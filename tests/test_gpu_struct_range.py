"""Structure functions of lbm_stats whose FP32 powers leave the FP32 range: infinite, as
plain sums of them are, and the lower powers unharmed."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(12, 14, 16), (30, 32, 36), (96, 104, 112)])
def test_powers_beyond_the_fp32_range(gpu_lib, shape):
    """Increments of 1e8: d^4 is 1e32, d^5 and d^6 are infinite.  d^2 of a cell carries 3
    roundings, its sum at most 4 x 4 more: 2e-6 is 32 x 2^-24."""
    lbm = gpu_lib
    nz, ny, nx = shape
    rng = np.random.default_rng(12)
    f = np.zeros((19, *shape))
    f[0] = rng.uniform(0.5e8, 1e8, size=shape)
    f[1] = -f[0]
    with lbm.Lattice(lbm.make_params(nx, ny, nz, nu0=0.01, cs=0.1, kernel=1, tile_rows=1, threads=128)) as L:
        L.set_populations(f)
        st = L.stats(what=lbm.LBM_STATS_STRUCTURE)
        u = L.fields()["u"]
    assert 1e7 < np.abs(u[0]).max() < 1e9
    for k, r in enumerate(st["r"]):
        d = np.concatenate([(np.roll(u[a], -r, axis=2 - a) - u[a]).ravel() for a in range(3)])
        for p in (2, 4):
            want = (d ** p).mean()
            assert abs(st["Sp"][k][p - 1] - want) <= 2e-6 * want
        assert np.isposinf(st["Sp"][k][5])

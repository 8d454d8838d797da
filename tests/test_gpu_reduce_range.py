"""Block reductions of the statistics at the ends of the FP32 range: sums that a warp
cannot hold in FP32, that are infinite already, or so small that low words would be
flushed, as FP64 sums of the same per-cell values give them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N = 16  # one cell per thread in every configuration below: no FP32 sum ahead of the reduction
CONFIGS = [dict(kernel=1, tile_rows=1, threads=64), dict(kernel=1, tile_rows=1, threads=256),
           dict(kernel=2, tile_rows=2, stages=3, threads=384)]


def _state(lbm, f, **cfg):
    L = lbm.Lattice(lbm.make_params(N, nu0=0.01, cs=0.13, **cfg))
    L.set_populations(f)
    return L


@pytest.mark.parametrize("cfg", CONFIGS)
def test_sums_beyond_the_fp32_range(gpu_lib, cfg):
    """|S|^2 of 2e38 a cell: 32 of them are beyond FP32, their FP64 mean is not; |S|^3 is
    infinite in each cell.  FP32 products of a cell carry a few roundings: 8 x 2^-24."""
    f = np.zeros((19, N, N, N))
    f[0], f[1] = 1e9, -1e9
    with _state(gpu_lib, f, **cfg) as L:
        st = L.stats()
        g = L.fields()
    tol = 8 * 2.0 ** -24
    ss = (g["snorm"] ** 2).mean()
    assert 1e38 < ss < 3.4e38
    assert abs(st["eps0"] - 0.01 * ss) <= tol * 0.01 * ss
    assert np.isposinf(st["eps_sgs"])
    uu = (g["u"] ** 2).sum(axis=0).mean()
    assert abs(st["E_k"] - 0.5 * uu) <= tol * uu
    assert abs(st["theta_mean"] - g["theta"].mean()) <= tol * g["theta"].mean()


@pytest.mark.parametrize("cfg", CONFIGS)
@pytest.mark.parametrize("scale", [1e-33, 1e-20, 1e-3])
def test_small_sums_keep_their_digits(gpu_lib, cfg, scale):
    """The mass is the FP64 sum of the cells' FP32 densities: 2^-45 of the sum of
    magnitudes (4096 terms, 2^-53 each)."""
    rng = np.random.default_rng(6)
    f = rng.normal(size=(19, N, N, N)) * scale
    with _state(gpu_lib, f, **cfg) as L:
        mass = L.stats()["mass"]
        drho = L.fields()["drho"]
    assert abs(mass - drho.sum()) <= 2.0 ** -45 * np.abs(drho).sum()

"""Block reductions of the statistics: sums whose lanes have, have not, or have partly
folded their FP32 sums into FP64 totals, against FP64 sums of the same fields; and the
statistics pass that gives up a stage of its pipeline for the theta histogram."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CONFIGS = [dict(kernel=1, tile_rows=1, threads=64), dict(kernel=1, tile_rows=1, threads=256),
           dict(kernel=2, tile_rows=2, stages=3, threads=384), dict(kernel=2, tile_rows=1, stages=2, threads=256, layout=2)]


@pytest.mark.parametrize("cfg", CONFIGS)
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 5, 7), (24, 20, 31), (100, 90, 110), (160, 152, 144)])
def test_sums_match_fields(gpu_lib, cfg, shape):
    """FP32 sums of at most 32 cells (one tile more on the TMA path) ahead of FP64:
    each carries at most 64 roundings, 64 x 2^-24 of the sum of magnitudes."""
    lbm = gpu_lib
    nz, ny, nx = shape
    rng = np.random.default_rng(2)
    u0 = rng.normal(scale=0.02, size=(3, *shape))
    p = lbm.make_params(nx, ny, nz, nu0=0.01, cs=0.13, f0=1e-4, force_mode=lbm.LBM_FORCE_PAPER_SIN, hist_max=0.2, **cfg)
    with lbm.Lattice(p) as L:
        L.init(lbm.LBM_INIT_VELOCITY, u=u0)
        L.step(3)
        st = L.stats()
        g = L.fields()
        h = lbm.lbm_histogram(L.h, 0, 4096)
    n, tol = nx * ny * nz, 64 * 2.0 ** -24
    u, th = g["u"], g["theta"]
    assert st["cells"] == n and int(h.sum()) == n
    q = th.astype(np.float32) * np.float32(4096 / 0.2)
    idx = np.where(q < 4096, np.floor(q), 4096).astype(np.int64)
    assert np.array_equal(h, np.bincount(idx.ravel(), minlength=4097))
    assert abs(st["mass"] - g["drho"].sum()) <= tol * np.abs(g["drho"]).sum()
    for k, (i, j) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
        assert abs(st["uu"][k] - (u[i] * u[j]).mean()) <= tol * np.abs(u[i] * u[j]).mean()
    for d in range(3):
        m = (1 + g["drho"]) * u[d]
        assert abs(st["momentum"][d] - m.sum()) <= tol * np.abs(m).sum()
    assert abs(st["theta_mean"] - th.mean()) <= tol * th.mean()
    assert abs(st["eps_sgs"] - 0.13 * (g["snorm"] ** 3).mean()) <= tol * 0.13 * (g["snorm"] ** 3).mean()
    assert st["theta_min"] == th.min() and st["theta_max"] == th.max()

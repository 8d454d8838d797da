"""The direct and the TMA step kernel give the same bits, so a handle's results do not
depend on which of them it runs: both strain modes, the storage types and layouts, plain
steps and steps with statistics, even and odd, and the read-only pass."""
import numpy as np
import pytest

from gpu_helpers import random_populations

pytestmark = pytest.mark.gpu

SHAPE = (17, 20, 32)  # nz, ny, nx
CONFIGS = [dict(kernel=1, tile_rows=1, threads=64), dict(kernel=1, tile_rows=1, threads=256, layout=2),
           dict(kernel=2, tile_rows=2, stages=2, threads=256), dict(kernel=2, tile_rows=3, stages=3, threads=384),
           dict(kernel=2, tile_rows=1, stages=4, threads=256, layout=2), dict(kernel=2, tile_rows=2, stages=2, threads=256, tma_slots=2)]


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("strain_mode", [0, 1])
@pytest.mark.parametrize("stats_every", [0, 1])
# at 0.000692 and 0.003267 the roundings of 1/2 + 3 nu0 differ with and without a fused step
@pytest.mark.parametrize("nu0", [0.01, 0.0003, 0.000692, 0.003267])
def test_bitwise(gpu_lib, precision, strain_mode, stats_every, nu0):
    nz, ny, nx = SHAPE
    f = random_populations(SHAPE, seed=3)
    want = None
    for cfg in CONFIGS:
        p = gpu_lib.make_params(nx, ny, nz, nu0=nu0, cs=0.16, f0=1e-4, force_mode=gpu_lib.LBM_FORCE_PAPER_SIN,
                                precision=precision, strain_mode=strain_mode, stats_every=stats_every, **cfg)
        with gpu_lib.Lattice(p) as L:
            L.set_populations(f)
            got = [L.fields()["theta"]]
            for steps in (1, 1, 7, 32):
                L.step(steps)
                got.append(L.populations())
            got.append(L.fields()["snorm"])
        want = want or got
        assert all(np.array_equal(a, b) for a, b in zip(got, want)), cfg

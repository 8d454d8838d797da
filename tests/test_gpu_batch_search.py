"""Batches whose instances a block of the direct kernel has to search: many alike, sizes that
mislead its guess, and the time a step of many small ones takes."""
import time

import numpy as np
import pytest

from gpu_helpers import random_populations

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes", [[(3, 5, 7)] * 40, [(1, 1, 1)] * 30 + [(12, 16, 20)] * 3, [(12, 16, 20)] * 2 + [(1, 2, 3)] * 40 + [(9, 10, 30)],
                                    [(2, 3, 4 + k) for k in range(60)]])
@pytest.mark.parametrize("threads", [64, 256])
def test_batch_steps_as_its_instances_alone(gpu_lib, shapes, threads):
    par = [gpu_lib.make_params(nx, ny, nz, nu0=0.01, cs=0.13, kernel=1, tile_rows=1, threads=threads) for nz, ny, nx in shapes]
    with gpu_lib.Lattice(par) as L:
        fs = [random_populations(s, seed=20 + i) for i, s in enumerate(shapes)]
        for i, f in enumerate(fs):
            L.set_populations(f, inst=i)
        L.step(5)
        for i in sorted({0, 1, len(shapes) // 2, len(shapes) - 2, len(shapes) - 1}):
            with gpu_lib.Lattice(par[i]) as one:
                one.set_populations(fs[i])
                one.step(5)
                assert np.array_equal(L.populations(inst=i), one.populations())


def _step_time(lbm, params):
    with lbm.Lattice(params) as L:
        L.step(64)
        L.sync()
        times = []
        for _ in range(9):
            t = time.perf_counter()
            L.step(128)
            L.sync()
            times.append(time.perf_counter() - t)
        return sorted(times)[4]


def test_many_instances_step_like_few(gpu_lib):
    """The same cells in 10 long boxes and in 200 cubes, 19 and 22 us a step; 51 when
    instances were gone through one by one.  The line lies between, far from the noise."""
    cfg = dict(nu0=0.01, cs=0.13, kernel=1, tile_rows=1, threads=128)
    many = _step_time(gpu_lib, [gpu_lib.make_params(16, **cfg) for _ in range(200)])
    few = _step_time(gpu_lib, [gpu_lib.make_params(16, 16, 320, **cfg) for _ in range(10)])
    assert many <= 1.8 * few, (many, few)

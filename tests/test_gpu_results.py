"""Results on their way to the host: outputs larger than a transfer chunk and than the size
from which pages are touched ahead, slices and records in several pieces, and errors that
arrive with the results."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_large_outputs(gpu_lib):
    """168^3: 4.7 M cells, so populations and fields go in two chunks per component; set
    and get are exact, the velocity is that of the fields, a slice is the fields' plane."""
    lbm = gpu_lib
    n = 168
    rng = np.random.default_rng(0)
    with lbm.Lattice(lbm.make_params(n, nu0=0.01, cs=0.1, kernel=1, tile_rows=1, threads=128)) as L:
        L.init_random(seed=2)
        L.step(3)
        f = L.populations()
        g = L.fields()
        v = lbm.lbm_get_velocity(L.h, 0, (n, n, n))
        assert np.array_equal(v, g["u"])
        for axis in range(3):
            assert np.array_equal(L.theta_slice(axis, 5), np.take(g["theta"], 5, axis=2 - axis))
        assert np.array_equal(f.sum(axis=0).astype(np.float32).shape, g["drho"].shape)
        assert np.max(np.abs(f.sum(axis=0) - g["drho"])) < 1e-6
        f2 = rng.permutation(f.reshape(19, -1), axis=1).reshape(f.shape)
        L.set_populations(f2)
        assert np.array_equal(L.populations(), f2)


def test_records_across_the_ring(gpu_lib):
    """More records than the ring holds, read in pieces: the last 1024, in order, each once,
    and the same as those of an identical run that reads one at a time."""
    lbm = gpu_lib
    params = [lbm.make_params(8, nu0=0.01, stats_every=1, kernel=1, tile_rows=1, threads=64),
              lbm.make_params(6, nu0=0.01, stats_every=1, kernel=1, tile_rows=1, threads=64)]

    def start():
        L = lbm.Lattice(params)
        L.init(lbm.LBM_INIT_TGV3D, amplitude=0.01, inst=0)
        L.init(lbm.LBM_INIT_TGV3D, amplitude=0.02, inst=1)
        return L

    with start() as L, start() as one:
        each = []
        for k in range(1500):
            one.step(1)
            each += lbm.lbm_series(one.h, 1, 4)
        assert [r["step"] for r in each] == list(range(1500))
        L.step(700)
        assert lbm.lbm_series(L.h, 1, 300) == each[:300]
        L.step(800)  # 1500 in all: 476 is the oldest the ring still holds
        assert lbm.lbm_series(L.h, 1, 1024) == each[476:]
        assert lbm.lbm_series(L.h, 1, 1024) == []
        assert len(lbm.lbm_series(L.h, 0, 5)) == 5


def test_errors_come_with_the_results(gpu_lib):
    """A non-finite cell: statistics, with and without the derived quantities, report it, a
    later spectrum is of the later state."""
    lbm = gpu_lib
    u = np.full((3, 12, 12, 12), 0.01)
    with lbm.Lattice(lbm.make_params(12, nu0=0.01, cs=0.1)) as L:
        bad = u.copy()
        bad[0, 3, 4, 5] = np.nan
        for what in (0, 3):
            L.init(lbm.LBM_INIT_VELOCITY, u=bad)
            with pytest.raises(lbm.LbmError) as ei:
                L.stats(what=what)
            assert ei.value.code == lbm.LBM_ERR_UNSTABLE
            L.init(lbm.LBM_INIT_VELOCITY, u=u)
            E = L.spectrum(3)
            assert abs(E[0] - 1.5e-4) < 1e-9 and np.all(E[1:] < 1e-12)
            assert L.stats(what=3)["cells"] == 12 ** 3

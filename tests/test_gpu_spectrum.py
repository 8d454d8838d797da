"""Energy spectrum: the framework's own transform and shell sums at the sizes
where they can go wrong (every radix, odd planes, one-cell extents, tiles with
ragged columns, long columns in narrow tiles), and the fallback for extents with
large prime factors, against numpy's FP64 transform of the same velocity."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _spectrum(u, kmax):
    _, nz, ny, nx = u.shape
    k = [np.abs(np.fft.fftfreq(n) * n).round() for n in (nz, ny, nx)]
    K = k[0][:, None, None] ** 2 + k[1][:, None] ** 2 + k[2] ** 2
    shell = np.floor(np.sqrt(K) + 0.5).astype(int)
    e = sum(np.abs(np.fft.fftn(u[d])) ** 2 for d in range(3)) * 0.5 / float(nx * ny * nz) ** 2
    E = np.bincount(shell.ravel(), e.ravel(), minlength=kmax + 1)
    return E[:kmax + 1]


def _max_shell(nx, ny, nz):
    return math.floor(math.sqrt((nx // 2) ** 2 + (ny // 2) ** 2 + (nz // 2) ** 2) + 0.5)


SHAPES = [  # nz, ny, nx
    (16, 16, 16), (10, 12, 18), (2, 3, 5), (1, 1, 1), (1, 8, 30), (7, 11, 13), (9, 15, 21), (13, 9, 25),  # odd planes
    (26, 22, 14), (100, 20, 24), (6, 250, 8), (8, 6, 1024), (1024, 4, 6), (4, 900, 10), (33, 50, 49),
    (17, 12, 20), (5, 19, 23), (6, 4, 1202), (37, 31, 29),  # cuFFT
]


@pytest.mark.parametrize("shape", SHAPES)
def test_spectrum_matches_fp64_transform(gpu_lib, shape):
    """FP32 transform: noise of 2^-24 per stage and point, log2 N stages; 1e-5 of
    a shell's energy plus 1e-9 of the total covers shells up to the tests' largest
    box (parity tests elsewhere allow 1e-4)."""
    lbm = gpu_lib
    nz, ny, nx = shape
    rng = np.random.default_rng(11)
    u0 = rng.normal(scale=0.03, size=(3, *shape))
    with lbm.Lattice(lbm.make_params(nx, ny, nz, nu0=0.01, cs=0.1)) as L:
        L.init(lbm.LBM_INIT_VELOCITY, u=u0)
        u = L.fields()["u"]
        kmax = _max_shell(nx, ny, nz)
        E = L.spectrum(kmax + 2)
        want = _spectrum(u, kmax)
        assert np.all(E[kmax + 1:] == 0.0)
        assert np.all(np.abs(E[:kmax + 1] - want) <= 1e-5 * want + 1e-9 * want.sum())
        L.step(2)  # another state, fewer shells
        low = kmax // 2
        want = _spectrum(L.fields()["u"], kmax)
        assert np.all(np.abs(L.spectrum(low) - want[:low + 1]) <= 1e-5 * want[:low + 1] + 1e-9 * want.sum())


def test_batch_and_chunked_components(gpu_lib):
    """A lattice whose three half spectra exceed one batch goes component by
    component: Parseval, and every shell against the batched size's rule (a field of
    one Fourier mode puts all its energy in that mode's shell)."""
    lbm = gpu_lib
    n, k = 320, 5
    x = np.sin(2 * np.pi * k * np.arange(n) / n)
    u0 = np.zeros((3, n, n, n), dtype=np.float32)
    u0[0] = 0.02 * x[:, None, None]  # varies along z
    u0[1] = 0.01 * x[None, None, :]
    u0[2] = 0.03 * x[None, :, None]
    with lbm.Lattice(lbm.make_params(n, nu0=0.01, kernel=1, tile_rows=4, threads=256)) as L:
        L.init(lbm.LBM_INIT_VELOCITY, u=u0)
        E = L.spectrum(40)
    total = 0.25 * (0.02 ** 2 + 0.01 ** 2 + 0.03 ** 2)
    assert abs(E[k] - total) <= 1e-5 * total
    assert np.sum(np.delete(E, k)) <= 1e-9 * total

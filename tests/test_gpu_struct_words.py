"""Structure functions of fields whose pencils repeat, in three-word sums: a rounding that
is the same in every run of cells adds up instead of averaging away."""
import numpy as np
import pytest

from test_gpu_struct import _noalloc, _sums

pytestmark = pytest.mark.gpu


def _field(kind, shape):
    nz, ny, nx = shape
    X, Y, Z = (2 * np.pi * np.arange(n) / n for n in (nx, ny, nz))
    X, Y, Z = X[None, None, :], Y[None, :, None], Z[:, None, None]
    one = np.ones(shape)
    if kind == "sine":    # u_x of x alone: every pencil along x alike
        u = [0.05 * np.sin(X) * one, 0 * one, 0 * one]
    elif kind == "sines":
        u = [0.05 * np.sin(X) * one, 0.04 * np.sin(Y) * one, 0.03 * np.sin(Z) * one]
    elif kind == "taylor_green":
        u = [0.05 * np.cos(X) * np.sin(Y) * np.sin(Z), -0.03 * np.sin(X) * np.cos(Y) * np.sin(Z),
             -0.02 * np.sin(X) * np.sin(Y) * np.cos(Z)]
    else:                 # constant gradient with one jump per pencil
        u = [0.001 * np.arange(n).reshape([-1 if a == d else 1 for d in range(3)]) / 3 * one
             for a, n in ((2, nx), (1, ny), (0, nz))]
    return np.array(u, dtype=np.float32)


@pytest.mark.parametrize("kind", ["sine", "sines", "taylor_green", "ramp"])
@pytest.mark.parametrize("shape", [(64, 64, 64), (24, 24, 128), (16, 18, 256), (40, 41, 47), (5, 33, 600)])
def test_repeated_pencils(gpu_lib, kind, shape):
    """All shapes are of 2^16 cells or more.  Beyond the words, whose roundings are below
    2^-60 of a sum, a sum takes at most 32 additions in FP64 (tiles of a block, its
    warps, the blocks): 32 x 2^-53 of the sum of |d|^p."""
    u, seps = _field(kind, shape), [1, 2, 5, 16]
    want, mag = _sums(u, seps)
    err = np.abs(_noalloc(gpu_lib, u, seps) - want)
    assert np.all(err <= 32 * 2.0 ** -53 * mag), np.max(err / np.where(mag > 0, mag, 1), axis=0)

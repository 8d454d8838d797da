"""Exact structure functions of fields whose increments are below the normal FP32 range
(flushed to zero in FP32 arithmetic, not in FP64), and of constant ones."""
import numpy as np
import pytest

from test_gpu_struct import _noalloc, _sums

pytestmark = pytest.mark.gpu

SEPS = [1, 3]


@pytest.mark.parametrize("shape", [(40, 41, 47), (8, 9, 40), (64, 64, 64)])
def test_subnormal_increments(gpu_lib, shape):
    """Normal values whose differences are subnormal; 1e-14 of the sum of |d|^p as for
    every other field."""
    rng = np.random.default_rng(9)
    u = (2e-38 * (1 + 0.3 * rng.random((3, *shape)))).astype(np.float32)
    want, mag = _sums(u, SEPS)
    assert np.all(mag[:, 1] > 1e-80)
    got = _noalloc(gpu_lib, u, SEPS)
    assert np.all(np.abs(got - want) <= 1e-14 * mag), (got, want)


@pytest.mark.parametrize("shape", [(40, 41, 47), (8, 9, 40)])
def test_zeros_of_either_sign(gpu_lib, shape):
    u = np.zeros((3, *shape), np.float32)
    u[:, ::2] *= -1
    u[1] = 0.25
    assert np.all(_noalloc(gpu_lib, u, SEPS) == 0.0)

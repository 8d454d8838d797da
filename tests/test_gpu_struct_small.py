"""Exact structure functions of small lattices, on fields whose pencils repeat: as far from
quadruple-precision sums as those of large ones."""
import numpy as np
import pytest

from test_gpu_struct import _noalloc, _sums
from test_gpu_struct_words import _field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["sine", "sines", "taylor_green", "ramp", "random"])
@pytest.mark.parametrize("shape", [(8, 8, 8), (16, 20, 24), (40, 40, 40), (7, 9, 500), (500, 9, 7), (2, 2, 2000)])
def test_small_lattices(gpu_lib, kind, shape):
    """A sum takes at most 32 additions in FP64 beyond the words: 32 x 2^-53 of the sum of
    |d|^p."""
    if kind == "random":
        u = np.random.default_rng(4).normal(scale=0.05, size=(3, *shape)).astype(np.float32)
    else:
        u = _field(kind, shape)
    seps = [1, 2, 3, 5]
    want, mag = _sums(u, seps)
    assert np.all(np.abs(_noalloc(gpu_lib, u, seps) - want) <= 32 * 2.0 ** -53 * mag)

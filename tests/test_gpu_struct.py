"""Structure functions: the tiled kernels at the edges of their tiles.

Pencils shorter and longer than a segment, extents that leave a tile's 32
pencils ragged, separations that wrap (also more than once) and ones too long
for a tile, values far outside the usual range.  The oracle is numpy in long
double on the same FP32 field.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _sums(u, seps):
    """<d^p> and <|d|^p> over cells and axes in long double, and the increments' sign kept."""
    n = u[0].size
    s, m = np.zeros((len(seps), 6)), np.zeros((len(seps), 6))
    v = u.astype(np.longdouble)
    for k, r in enumerate(seps):
        d = np.concatenate([(np.roll(v[a], -(r % u.shape[3 - a]), axis=2 - a) - v[a]).ravel() for a in range(3)])
        p = d.copy()
        for q in range(6):
            s[k, q] = np.sum(p) / (3 * n)
            m[k, q] = np.sum(np.abs(p)) / (3 * n)
            p *= d
    return s, m


def _noalloc(lbm, u, seps):
    import torch
    dev = torch.device("cuda", 0)
    sp = torch.full((len(seps), 6), float("nan"), dtype=torch.float64, device=dev)
    lbm.lbm_structure_functions_noalloc(torch.from_numpy(u).to(dev), seps, sp)
    torch.cuda.synchronize()
    return sp.cpu().numpy()


SHAPES = [  # nz, ny, nx: extents of 1 and 2, one cell past a segment, past two of them, ragged pencils
    ((1, 2, 33), [1, 2, 3]),
    ((31, 5, 7), [1, 4, 40]),
    ((6, 257, 9), [1, 128, 256]),
    ((20, 3, 513), [1, 2, 3, 256, 512]),
    ((1030, 5, 4), [7, 500, 1029, 3000]),
    ((33, 40, 64), list(range(1, 25))),
    ((2, 3, 3000), [1, 1900]),  # 1900 cells do not fit a tile
    ((41, 43, 47), [1, 2, 5, 20]),  # above the size from which terms are kept in FP32 words
    ((5, 1100, 33), [3, 400, 600]),
]


@pytest.mark.parametrize("shape,seps", SHAPES)
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -50, 2.0 ** 50])
def test_fp64_sums_of_a_device_field(gpu_lib, shape, seps, scale):
    """FP64 accuracy: 1e-14 of the sum of |d|^p allows 2^6 FP64 roundings."""
    rng = np.random.default_rng(7)
    u = (rng.normal(scale=0.05, size=(3, *shape)) * scale).astype(np.float32)
    want, mag = _sums(u, seps)
    got = _noalloc(gpu_lib, u, seps)
    assert np.all(np.abs(got - want) <= 1e-14 * mag + 0.0), np.max(np.abs(got - want) / np.where(mag > 0, mag, 1))


def test_values_outside_the_scaled_range(gpu_lib):
    """Zero, constant and huge fields, and non-finite cells, as FP64 gives them."""
    shape, seps = (8, 9, 40), [1, 3]
    assert np.all(_noalloc(gpu_lib, np.zeros((3, *shape), np.float32), seps) == 0.0)
    assert np.all(_noalloc(gpu_lib, np.full((3, *shape), 3.0e7, np.float32), seps) == 0.0)
    rng = np.random.default_rng(3)
    for scale in (1e30, 1e-30):
        u = (rng.normal(size=(3, *shape)) * scale).astype(np.float32)
        want, mag = _sums(u, seps)
        assert np.all(np.abs(_noalloc(gpu_lib, u, seps) - want) <= 1e-14 * mag)
    u = rng.normal(size=(3, *shape)).astype(np.float32)
    u[0, 2, 3, 4] = np.inf
    got = _noalloc(gpu_lib, u, seps)
    assert np.all(np.isposinf(got[:, 1::2])) and np.all(np.isnan(got[:, 0::2]))
    u[0, 2, 3, 4] = np.nan
    assert np.all(np.isnan(_noalloc(gpu_lib, u, seps)))


@pytest.mark.parametrize("shape", [(3, 4, 5), (20, 33, 31), (12, 14, 300), (40, 530, 36)])
def test_statistics_agree_with_fp64_sums(gpu_lib, shape):
    """lbm_stats: FP32 increments and powers.  A power carries at most 7
    roundings, a warp's sum of 64 cells and 32 lanes at most 64 + 5: 80 x 2^-24
    of the sum of |d|^p (the roundings of one sum do not all point one way)."""
    lbm = gpu_lib
    nz, ny, nx = shape
    rng = np.random.default_rng(5)
    u0 = rng.normal(scale=0.03, size=(3, *shape))
    with lbm.Lattice(lbm.make_params(nx, ny, nz, nu0=0.01, cs=0.1)) as L:
        L.init(lbm.LBM_INIT_VELOCITY, u=u0)
        L.step(2)
        st = L.stats(what=lbm.LBM_STATS_STRUCTURE)
        u = L.fields()["u"].astype(np.float32)
    want, mag = _sums(u, st["r"])
    assert np.all(np.abs(st["Sp"] - want) <= 80 * 2.0 ** -24 * mag)

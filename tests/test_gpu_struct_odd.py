"""Structure functions of lbm_stats on a smooth field: neighbouring increments are alike,
so long plain FP32 sums of odd powers, which cancel over a pencil, would lose digits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N = 256


def test_odd_powers_of_a_smooth_field(gpu_lib):
    """Plain FP32 sums span 4 cells.  One rounding has a standard deviation of at most 2^-24 / sqrt 3
    of the partial sum; alike increments make that up to k |d| after k cells, a variance
    of (1 + 4 + 9 + 16) / 4 = 7.5 a cell, and that of d is in its power p times: p^2.  Six
    standard deviations over the 3 N^3 cells, relative to the sum of |d|^p; rms over mean
    of |d|^p as for Gaussian increments."""
    import torch

    lbm = gpu_lib
    with lbm.Lattice(lbm.make_params(N, nu0=0.01, cs=0.1, kernel=1, tile_rows=1, threads=128)) as L:
        L.init_random(seed=5)
        L.step(2)
        st = L.stats(what=lbm.LBM_STATS_STRUCTURE)
        u = torch.from_numpy(L.fields()["u"].astype(np.float32)).cuda()
    one = 6 * 2.0 ** -24 / np.sqrt(3) / np.sqrt(3 * N ** 3)
    for k, r in enumerate(st["r"]):
        s, m = np.zeros(6), np.zeros(6)
        for a in range(3):
            v = u[a].double()
            d = torch.roll(v, -r, 2 - a) - v
            p = d.clone()
            for q in range(6):
                s[q] += float(p.sum()) / (3 * N ** 3)
                m[q] += float(p.abs().sum()) / (3 * N ** 3)
                p *= d
        for q, ratio in ((0, 1.26), (2, 2.43), (4, 4.82)):
            assert abs(st["Sp"][k][q] - s[q]) <= ratio * one * np.sqrt(7.5 + (q + 1) ** 2) * m[q], (r, q + 1)

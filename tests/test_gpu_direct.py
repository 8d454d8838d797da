"""The direct-load step kernel where its chunks of cells end: lattices smaller than a
block, chunks that run past an instance, every block size, both layouts and storage
widths, batches whose instances change within a block's walk, arrays of 4 GB and
more (64-bit offsets); and the dependent launches of consecutive steps."""
import numpy as np
import pytest

import oracle
from gpu_helpers import full_f_rel_error, random_populations, ulp

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (1, 2, 3), (3, 5, 7), (2, 33, 31), (13, 8, 20), (16, 16, 16)]  # nz, ny, nx
NU0, C, F0 = 0.01, 0.13, 1e-4


def _params(lbm, shape, threads, **kw):
    nz, ny, nx = shape
    return lbm.make_params(nx, ny, nz, nu0=NU0, cs=C, f0=F0, force_mode=lbm.LBM_FORCE_PAPER_SIN, kernel=1,
                           tile_rows=1, threads=threads, **kw)


def _reference(shape, f, steps):
    nz, ny, nx = shape
    ref = oracle.OracleLBM(nx, ny, nz, NU0, C, oracle.FORCE_PAPER_SIN, F0=F0)
    ref.set_populations(f)
    ref.step(steps)
    return ref.populations()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("threads", [64, 128, 256])
@pytest.mark.parametrize("layout,precision", [(1, 0), (2, 0), (1, 1), (2, 2)])
def test_direct_kernel_matches_oracle(gpu_lib, shape, threads, layout, precision):
    """FP32: 1e-5 relative (the parity bound); 16 bits: one spacing of the largest
    |f'| per step."""
    f = random_populations(shape, seed=4)
    steps = 37  # 32 replayed from a graph, then 5 launches
    want = _reference(shape, f, steps)
    with np.errstate(all="ignore"):
        with gpu_lib.Lattice(_params(gpu_lib, shape, threads, layout=layout, precision=precision)) as L:
            L.set_populations(f)
            L.step(steps)
            got = L.populations()
    if precision == 0:
        assert full_f_rel_error(got, want) < 1e-5
    else:
        top = max(np.max(np.abs(f)), np.max(np.abs(want)))
        assert np.max(np.abs(got - want)) <= (steps + 1) * ulp(top, 10 if precision == 1 else 7)


@pytest.mark.parametrize("threads", [64, 256])
def test_direct_kernel_batch_and_statistics(gpu_lib, threads):
    """Uneven instances in one launch, and the sums of the fused statistics over them."""
    shapes = [(1, 1, 1), (3, 5, 7), (2, 33, 31), (1, 2, 3), (9, 10, 11)]
    fs = [random_populations(s, seed=10 + i) for i, s in enumerate(shapes)]
    with gpu_lib.Lattice([_params(gpu_lib, s, threads, stats_every=3) for s in shapes]) as L:
        for i, f in enumerate(fs):
            L.set_populations(f, inst=i)
        L.step(7)
        for i, s in enumerate(shapes):
            assert full_f_rel_error(L.populations(inst=i), _reference(s, fs[i], 7)) < 1e-5
            rec = L.series(inst=i)
            assert [r["step"] for r in rec] == [0, 3, 6]
            # mass: sum of drho, conserved; each record against the FP64 sum of the input
            mass = fs[i].sum()
            assert all(abs(r["mass"] - mass) <= 1e-5 * max(1.0, np.abs(fs[i]).sum()) for r in rec)


def test_arrays_of_four_gigabytes(gpu_lib):
    """64-bit offsets: 388 x 384 x 384 cells (4.35 GB in FP32), an even and an odd step
    against the TMA kernel on every cell (the two kernels agree to 1e-7 of the
    largest |f'| per step)."""
    import torch

    lbm = gpu_lib
    out = []
    for cfg in (dict(kernel=1, tile_rows=1, threads=128), dict(kernel=2, tile_rows=1, stages=2, threads=256)):
        p = lbm.make_params(388, 384, 384, nu0=NU0, cs=C, f0=F0, force_mode=lbm.LBM_FORCE_PAPER_SIN, layout=1, **cfg)
        L = lbm.Lattice(p)
        L.init_random(seed=3)
        L.step(4)
        L.sync()
        ptr, nbytes, _ = lbm.lbm_device_ptr(L.h)
        assert nbytes >= 1 << 32

        class A:
            __cuda_array_interface__ = {"shape": (nbytes // 4,), "typestr": "<f4", "data": (ptr, False), "version": 3,
                                        "strides": None}
        out.append((L, torch.as_tensor(A(), device="cuda")))
    top = float(out[0][1].abs().max())
    worst = max(float((a - b).abs().max()) for a, b in zip(out[0][1].split(1 << 28), out[1][1].split(1 << 28)))
    assert worst <= 4e-7 * max(1.0, top)
    for L, _ in out:
        L.close()

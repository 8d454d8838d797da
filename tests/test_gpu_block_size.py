"""lbm_params.threads of a handle that asks for the direct kernel."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 40])
@pytest.mark.parametrize("threads", [64, 96, 128, 256])
def test_block_size_is_the_callers(gpu_lib, n, threads):
    with gpu_lib.Lattice(gpu_lib.make_params(n, nu0=0.01, kernel=1, threads=threads)) as L:
        assert L.config()["kind"] == 1 and L.config()["threads"] == threads


def test_blocks_beyond_the_launch_bound(gpu_lib):
    """Left to the autotuner, as ever."""
    with gpu_lib.Lattice(gpu_lib.make_params(8, nu0=0.01, kernel=1, threads=512)) as L:
        assert L.config()["kind"] == 1 and L.config()["threads"] <= 256
        L.init(gpu_lib.LBM_INIT_TGV3D, amplitude=0.02)
        L.step(3)
        assert L.stats()["cells"] == 512


@pytest.mark.parametrize("n", [48, 64, 80])
@pytest.mark.parametrize("stats_every", [1, 100])
def test_frequent_statistics_keep_larger_blocks(gpu_lib, n, stats_every):
    """A step with statistics reduces per block: 64 threads cost it 10 us over 128."""
    with gpu_lib.Lattice(gpu_lib.make_params(n, nu0=0.01, cs=0.13, stats_every=stats_every)) as L:
        assert L.config()["kind"] == 2 or L.config()["threads"] >= 128

"""Lattices of many small planes: a TMA tile never crosses one, so the direct kernel steps
them 1.5 times and more as fast, and the autotuner has to find that."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_a_long_box(gpu_lib, precision):
    with gpu_lib.Lattice(gpu_lib.make_params(8, 8, 30000, nu0=0.01, cs=0.13, precision=precision)) as L:
        assert L.config()["kind"] == 1


def test_a_batch_of_small_boxes(gpu_lib):
    with gpu_lib.Lattice([gpu_lib.make_params(16, nu0=0.01, cs=0.13) for _ in range(200)]) as L:
        assert L.config()["kind"] == 1

"""The kernels with index arithmetic of their own under the bounds-checked build: ragged chunks
and 32-bit offsets of the direct kernel, every radix and odd planes of the transform,
wrapped halos and short segments of the structure functions, the block reductions and
the results on their way to the host.  Their tests run against that build in a child
process and pass unchanged: no access out of bounds."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FILES = ["direct", "spectrum", "struct", "struct_long", "struct_small", "struct_range", "struct_underflow",
         "reduce", "reduce_range", "results", "slices", "outputs"]


def test_kernels_under_the_checked_build(gpu_lib):
    env = dict(os.environ, LBM_LIBRARY="checked")
    # (one file compares times, which the checks lengthen)
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider", "-k", "not takes_no_longer",
                        *[f"tests/test_gpu_{f}.py" for f in FILES]],
                       cwd=ROOT, env=env, capture_output=True, text=True, timeout=1800)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
    assert " passed" in r.stdout

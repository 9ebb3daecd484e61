"""The hardware forms that stand for CUDA's own functions: the same bits over the
ranges they are used in, and the FP64 reciprocal square root within its bound."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu


def test_forms_against_cuda_functions(tmp_path):
    from paper_2608_14544_gb300 import build

    exe = str(tmp_path / "forms")
    src = os.path.join(os.path.dirname(__file__), "approx_forms.cu")
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, src, "-o", exe],
                   check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    rsqrt, rcp, div, pairs = map(int, out[:4])
    assert pairs > 1 << 28
    assert (rsqrt, rcp, div) == (0, 0, 0)
    # in units of 2^-53: a half for each of the rounded x y (as an error of e, of
    # which half reaches y), the sum e y (...) + y, and what the seed and the series
    # leave (far below); and one for the last place of a y just above a power of two
    assert float(out[4]) <= 2.0

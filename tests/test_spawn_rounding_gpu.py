"""The FP32 spawning test is evaluated in several places (counted for the next
step, taken, and again for the child's weight), so its bits must not depend on
how each copy is compiled: built with and without multiply-add contraction it
gives the same thresholds, events, amplitudes and child weights."""
import os
import subprocess
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_bits_do_not_depend_on_contraction(tmp_path):
    from paper_2608_14544_gb300 import build

    src = os.path.join(os.path.dirname(__file__), "spawn_rounding.cu")

    def compiled(fmad):
        exe = str(tmp_path / f"fmad_{fmad}")
        subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC,
                        f"-fmad={fmad}", src, "-o", exe], check=True)
        return exe

    with ThreadPoolExecutor(2) as pool:
        exes = list(pool.map(compiled, ("true", "false")))
    rec = np.dtype([("T", "u4"), ("ev", "u4"), ("deg", "u4"), ("fac", "u4"), ("hi", "u4"),
                    ("lo", "u4"), ("ph", "u4"), ("e", "i4")])
    a, b = (np.frombuffer(subprocess.run([e], check=True, capture_output=True).stdout, rec)
            for e in exes)
    assert a.size == b.size == 4 << 18
    for form in range(4):
        x, y = (v[form << 18:(form + 1) << 18] for v in (a, b))
        assert 1000 < np.count_nonzero(x["ev"]) < x.size
        for key in rec.names:
            assert np.array_equal(x[key], y[key]), (form, key)

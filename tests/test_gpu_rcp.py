"""The packed kernels' reciprocal (neg_rcp2) against CUDA's correctly rounded one, over all FP32
values in either half of a pair: k_step2 and k_resident have the bits of k_step only if these agree."""
import os
import subprocess

import pytest

from paper_1008_2865_gb300 import build as lbbuild

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_neg_rcp2_is_the_rounded_reciprocal_everywhere(tmp_path):
    exe = str(tmp_path / "rcp_check")
    subprocess.run([lbbuild._nvcc(), *lbbuild.ARCH, "-O3", "-std=c++17", "-I" + lbbuild.INCLUDE,
                    "-I" + lbbuild.CSRC, os.path.join(ROOT, "tests", "c", "rcp_check.cu"), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout

"""The square root and quotient of the voxel-grid form (Markstein's Newton steps on the
reciprocal root) against CUDA's correctly rounded operations: all 2^23 mantissas at the
exponents of their domain that squared distances take (ROOT_MIN = 2^-96, to which the
kernel raises smaller ones, to 2^30), eight quotients for each.  No result may differ."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_1804_06304_gb300 import build
    exe = str(tmp_path_factory.mktemp("probe") / "root_quotient")
    subprocess.run([build.NVCC, *build.ARCH, "-O3", "-std=c++17", "-I" + build.INCLUDE, "-o", exe,
                    os.path.join(HERE, "_root_quotient_ref.cu")], check=True, capture_output=True)
    return exe


@pytest.mark.parametrize("first,last", [(-96, -60), (-59, -11), (-10, 30)])
def test_roots_and_quotients_are_correctly_rounded(probe, first, last):
    out = subprocess.run([probe, str(first), str(last)], check=True, capture_output=True, text=True, timeout=120)
    assert out.stdout.split() == ["0", "0"]

"""One block of the decimation's singular vectors: limits that are refused."""
import ctypes as C
import os
import subprocess

import pytest

from paper_1703_04789_gb300 import build as B
from tests.gpu_util import gpu_available

INVALID_VALUE = 1  # cudaErrorInvalidValue


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("svd") / "libsvd_unit.so")
    here = os.path.dirname(os.path.abspath(__file__))
    subprocess.run([B._nvcc(), "-std=c++17", "-O2", *B.ARCH, "-shared", "-Xcompiler", "-fPIC", "-I", B.CSRC, "-o", out,
                    os.path.join(here, "svd_unit.cu"), os.path.join(B.CSRC, "svd.cu")], check=True, capture_output=True)
    return C.CDLL(out)


@pytest.mark.parametrize("dim,other", [(1025, 1025), (2000, 4000)])
def test_blocks_beyond_the_limits_are_refused(lib, dim, other):
    if gpu_available():
        pytest.skip("shown without a device: a launch would need one")
    assert lib.svd_launch_empty(dim, other) == INVALID_VALUE

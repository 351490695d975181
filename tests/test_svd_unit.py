"""One block of the decimation's singular vectors: limits that are refused, sweeps that end too early.

Singular values of a block of norm 1 are FP64 rounding of it: 1e-14 for some hundreds of rows (a few n eps); the
vectors' orthonormality 1e-12, as in the tests of the canonical form.
"""
import ctypes as C
import os
import subprocess

import numpy as np
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


@pytest.mark.parametrize("dim,other,sweeps", [(1025, 1025, 250), (2000, 4000, 250), (8, 8, 257)])
def test_blocks_beyond_the_limits_are_refused(lib, dim, other, sweeps):
    if gpu_available():
        pytest.skip("shown without a device: a launch would need one")
    assert lib.svd_launch_empty(dim, other, sweeps) == INVALID_VALUE


def _block(lib, x, sweeps=250):
    dim, other = x.shape
    ev, vec, flag = np.empty(dim), np.empty((dim, dim)), C.c_int(-1)
    ptr = lambda a: a.ctypes.data_as(C.POINTER(C.c_double))
    assert lib.svd_block(dim, other, sweeps, ptr(x), ptr(ev), ptr(vec), C.byref(flag)) == 0
    return np.sqrt(np.maximum(ev, 0.0)), vec, flag.value


@pytest.mark.gpu
@pytest.mark.parametrize("dim,other", [(1, 3), (9, 9), (100, 25), (25, 100), (130, 150), (300, 300)])
def test_block_reports_whether_it_settled(lib, dim, other):
    if not gpu_available():
        pytest.skip("needs a CUDA device")
    x = np.random.default_rng(dim).standard_normal((dim, other))
    x /= np.linalg.norm(x)
    k = min(dim, other)
    # one sweep leaves couplings where two rows or more have a norm (a single row has none)
    assert _block(lib, x, 1)[2] == (1 if k > 1 else 0)
    values, vec, flag = _block(lib, x)
    assert flag == 0
    assert np.abs(values[:k] - np.linalg.svd(x, compute_uv=False)).max() < 1e-14
    assert np.abs(vec[:, :k].T @ vec[:, :k] - np.eye(k)).max() < 1e-12


@pytest.mark.gpu
def test_slowest_blocks_settle(lib):
    """Rows that differ little beside a few large columns need the most sweeps."""
    if not gpu_available():
        pytest.skip("needs a CUDA device")
    rng = np.random.default_rng(0)
    x = rng.standard_normal((400, 500)) * 10.0 ** -rng.uniform(0, 14, 400)[:, None]
    assert _block(lib, x / np.linalg.norm(x))[2] == 0


@pytest.mark.gpu
@pytest.mark.parametrize("dim,other", [(8, 40), (20, 40), (60, 100), (126, 250), (180, 300)])
def test_vectors_are_orthonormal_to_rounding(lib, dim, other):
    """Blocks whose vectors are the accumulated rotations, singular values over 14 decades: a rotation moves the
    product of two rows by at most four roundings, and a row takes part in dim rotations of each of up to 20 sweeps."""
    if not gpu_available():
        pytest.skip("needs a CUDA device")
    rng = np.random.default_rng(dim)
    u, v = (np.linalg.qr(rng.standard_normal((n, dim)))[0] for n in (dim, other))
    x = (u * 10.0 ** -np.linspace(0, 14, dim)) @ v.T
    _, vec, flag = _block(lib, x / np.linalg.norm(x))
    assert flag == 0
    assert np.abs(vec.T @ vec - np.eye(dim)).max() < 4 * 2.0 ** -53 * np.sqrt(20 * dim)


@pytest.mark.gpu
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("dim,other", [(60, 100), (100, 60), (160, 200)])
def test_block_that_overflowed_has_no_values(lib, bad, dim, other):
    if not gpu_available():
        pytest.skip("needs a CUDA device")
    x = np.random.default_rng(dim).standard_normal((dim, other))
    x[dim // 2, other // 3] = bad
    values, _, flag = _block(lib, x)
    assert flag == 0 and not values.any()


@pytest.mark.gpu
def test_state_that_overflows_is_an_error():
    if not gpu_available():
        pytest.skip("needs a CUDA device")
    from paper_1703_04789_gb300 import Spmps, SpmpsError, inputs
    labels, tens = inputs.random_mps(6, 6, 0, 16, 1)
    dev = Spmps(6, 6, 0, 0, 4, 16)
    dev.set_hubbard(1.0, 4.0)
    dev.set_mps(labels, tens, center=0)
    dev.canonicalize()
    dev.set_mps(labels, tens[:4] + [tens[4] * 1e200, tens[5] * 1e200], center=0)
    with pytest.raises(SpmpsError):
        dev.canonicalize()
    dev.close()

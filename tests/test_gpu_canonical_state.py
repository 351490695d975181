"""The canonical form is that of the same state, for states whose singular values fall over many decades.

The overlap is taken on the host.  A singular value below 1e-7 of the norm is dropped: at most 4 D of them at
each of the K - 1 bonds, 1e-14 of the squared norm each, and 1 - overlap is at most their sum.
"""
import numpy as np
import pytest

from paper_1703_04789_gb300 import inputs
from tests.gpu_util import require_gpu


def _overlap(A, B):
    E = np.ones((1, 1))
    for a, b in zip(A, B):
        E = np.einsum("bsc,bsd->cd", np.einsum("ab,asc->bsc", E, a), b)
    return float(E[0, 0])


@pytest.mark.gpu
@pytest.mark.parametrize("K,D,smem_max", [(7, 24, 0), (8, 90, 0), (8, 90, 8), (10, 150, 0)])
@pytest.mark.parametrize("graded", [(), (1, 2, 4), (1, 2, 3, 4, 5)])
def test_canonical_form_is_the_same_state(K, D, smem_max, graded):
    require_gpu()
    from paper_1703_04789_gb300 import Spmps
    labels, tens = inputs.random_mps(K, 6, 0, D, 3)
    for i in graded:
        tens[i] = tens[i] * 10.0 ** -((7 * np.arange(tens[i].shape[2])) % 13)
    dev = Spmps(K, 6, 0, 0, 4, D, jacobi_smem_max=smem_max)
    dev.set_hubbard(1.0, 4.0)
    dev.set_mps(labels, tens, center=0)
    dev.canonicalize()
    _, ts, _ = dev.get_mps()
    dev.close()
    tens = [t / np.linalg.norm(t) for t in tens]
    ov = _overlap(tens, ts) / np.sqrt(_overlap(tens, tens) * _overlap(ts, ts))
    assert 1.0 - abs(ov) <= (K - 1) * 4 * D * 1e-14

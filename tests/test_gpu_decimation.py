"""Singular vectors of the decimation (one-sided Jacobi, FP32 start, FP64 finish).

Canonicalising a raw state runs one decimation per bond with blocks of every shape: more rows than
columns and the other way round, rank-deficient ones, single rows.  Afterwards every site right of the
centre is an isometry and the state is the same.  The bounds are FP64 rounding: an isometry of n rows
deviates by a few n eps (1e-12 for n up to 200), the energy by 1e-10 as in the other parity tests.
"""
import numpy as np
import pytest

from oracle import mpo as M, mps as S
from paper_1703_04789_gb300 import inputs
from tests.gpu_util import require_gpu


def _deviation(labels, tensors):
    worst = 0.0
    for A in tensors[1:]:
        B = A.reshape(A.shape[0], -1)
        worst = max(worst, np.abs(B @ B.T - np.eye(B.shape[0])).max())
    return worst


@pytest.mark.gpu
@pytest.mark.parametrize("K,N,twoM,D,smem_max", [
    (4, 4, 0, 3, 0),        # single rows
    (7, 6, 0, 40, 0),       # ragged blocks
    (7, 6, 0, 40, 8),       # blocks above 8 start in global memory
    (8, 8, 0, 200, 0),      # up to the exact ranks: rank-deficient blocks at both ends
    (8, 5, 1, 330, 0),      # every Schmidt state kept
])
def test_canonical_form_is_isometric_and_keeps_the_state(K, N, twoM, D, smem_max):
    require_gpu()
    from paper_1703_04789_gb300 import Spmps
    labels, tens = inputs.random_mps(K, N, twoM, D, 3)
    P = S.prepare(labels, tens, M.hubbard_mpo(K, 1.0, 4.0), abs(twoM), twoM, 4)
    E_ref, nP_ref = P.energy(0)
    dev = Spmps(K, N, twoM, abs(twoM), 4, D, jacobi_smem_max=smem_max)
    dev.set_hubbard(1.0, 4.0)
    dev.set_mps(labels, tens, center=0)
    dev.canonicalize()
    lab, ts, c = dev.get_mps()
    assert c == 0 and all(t.shape[0] <= max(D, 1) for t in ts)
    assert _deviation(lab, ts) < 1e-12
    E, nP = dev.energy()
    assert abs(E - E_ref) < 1e-10 * max(1.0, abs(E_ref)) and abs(nP - nP_ref) < 1e-10
    dev.close()


@pytest.mark.gpu
@pytest.mark.parametrize("K,D,smem_max", [(7, 24, 0), (8, 90, 0), (8, 90, 8)])
def test_graded_states_stay_isometric(K, D, smem_max):
    """Singular values over twelve decades, most of a block's rows far below the largest: the rotation of two
    rows of very different norms, rows at the rounding noise, and values dropped below 1e-7."""
    require_gpu()
    from paper_1703_04789_gb300 import Spmps
    labels, tens = inputs.random_mps(K, 6, 0, D, 3)
    for i in (1, 2, 4):
        tens[i] = tens[i] * 10.0 ** -((7 * np.arange(tens[i].shape[2])) % 13)
    dev = Spmps(K, 6, 0, 0, 4, D, jacobi_smem_max=smem_max)
    dev.set_hubbard(1.0, 4.0)
    dev.set_mps(labels, tens, center=0)
    dev.canonicalize()
    lab, ts, _ = dev.get_mps()
    assert _deviation(lab, ts) < 1e-12
    dev.close()


@pytest.mark.gpu
def test_blocks_beyond_shared_memory_in_both_directions():
    """Blocks of up to 272 x 272, whose [Z | I] no longer fits one CTA's shared memory: canonicalisation
    (vectors of the right side), then steps to the right with one Davidson iteration each (the Ritz
    vector of a one-vector basis is the current two-site tensor, so the decimation only moves the gauge)."""
    require_gpu()
    from paper_1703_04789_gb300 import Spmps
    K, N, D = 12, 12, 700
    labels, tens = inputs.random_mps(K, N, 0, D, 5)
    dev = Spmps(K, N, 0, 0, 2, D, dav_max_iter=1)
    dev.set_hubbard(1.0, 4.0)
    dev.set_mps(labels, tens, center=0)
    E0, _ = dev.energy()  # a quotient: <P> of a state that is not canonical has no meaning
    dev.canonicalize()
    lab, ts, _ = dev.get_mps()
    assert _deviation(lab, ts) < 1e-12
    E1, _ = dev.energy()
    assert abs(E1 - E0) < 1e-10 * max(1.0, abs(E0))
    for k in range(6):
        dev.optimize_step(k, True, allow_not_converged=True)
    lab, ts, c = dev.get_mps()
    assert c == 6
    for A in ts[:6]:
        B = A.reshape(-1, A.shape[2])
        assert np.abs(B.T @ B - np.eye(B.shape[1])).max() < 1e-12
    E2, _ = dev.energy()
    assert abs(E2 - E0) < 1e-9 * max(1.0, abs(E0))
    dev.close()

"""The MPO-leg combination on unrotated operators: fused and separate forms, shared and own T1.

An action that wants both outputs reads N's T1 out of H's channel of identities where the operator has
one; an operator whose first two sites are scaled by 2 and 1/2 has none, but is the same operator.  All
forms are compared with the oracle (bound 1e-10 of the largest entry, as the other FP64 parity tests:
the forms differ from it only in summation order).
"""
import numpy as np
import pytest

from oracle import mpo as M, mps as S
from paper_1703_04789_gb300 import inputs
from tests.gpu_util import masked_random_two_site, require_gpu


def _ab_initio(K):
    h1, eri, _ = inputs.synthetic_active_space(K, 7)
    from paper_1703_04789_gb300 import mpo_from_integrals
    return mpo_from_integrals(h1, eri, 0.0)


@pytest.mark.gpu
@pytest.mark.parametrize("K,N,twoM,twoS,D,G,ab", [
    (2, 2, 0, 0, 4, 1, False),     # one pair, no environment on either side
    (6, 5, 1, 3, 13, 3, False),    # odd filling, at most 28 inputs per class: fused form
    (5, 4, 2, 2, 11, 2, True),     # hundreds of terms: separate rotation and combination
    (6, 9, 1, 1, 17, 3, True),     # nearly full band: labels missing on one side
])
@pytest.mark.parametrize("chain", [True, False])
def test_forms_match_oracle_and_each_other(K, N, twoM, twoS, D, G, ab, chain):
    require_gpu()
    from paper_1703_04789_gb300 import Spmps
    sites = [w.copy() for w in (_ab_initio(K) if ab else M.hubbard_mpo(K, 1.0, 3.0))]
    labels, tens = inputs.random_mps(K, N, twoM, D, 4)
    P = S.prepare(labels, tens, sites, twoS, twoM, G)
    if not chain:
        sites[0] *= 2.0
        sites[1] *= 0.5
    dev = Spmps(K, N, twoM, twoS, G, D)
    dev.set_mpo(sites)
    dev.set_mps(P.mps.labels, P.mps.A, center=0)
    one = Spmps(K, N, twoM, twoS, G, D, batched=False)
    one.set_mpo(sites)
    one.set_mps(P.mps.labels, P.mps.A, center=0)
    import torch
    P.build_left(K - 2)
    rng = np.random.default_rng(1)
    for k in range(K - 1):
        ql, qr = P.mps.labels[k], P.mps.labels[k + 2]
        lay = dev.x_layout(k)
        x = masked_random_two_site(ql, qr, rng)
        xv = dev.pack(x, lay, ql, qr)
        y, z = dev.apply_heff_host(k, xv)
        y_ref, z_ref = P.apply(x, k)
        assert np.abs(dev.unpack(y, lay, ql, qr) - y_ref).max() <= 1e-10 * max(1.0, np.abs(y_ref).max())
        assert np.abs(dev.unpack(z, lay, ql, qr) - z_ref).max() <= 1e-10 * max(1.0, np.abs(z_ref).max())
        # each output alone, and beta point by beta point: the same numbers
        t = torch.tensor(xv, device="cuda")
        a, b = torch.empty_like(t), torch.empty_like(t)
        dev.apply_heff(k, t, a, None)
        dev.apply_heff(k, t, None, b)
        torch.cuda.synchronize()
        y1, z1 = one.apply_heff_host(k, xv)
        assert np.array_equal(a.cpu().numpy(), y) and np.array_equal(b.cpu().numpy(), z)
        assert np.array_equal(y1, y) and np.array_equal(z1, z)
    dev.close()
    one.close()

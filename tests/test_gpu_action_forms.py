"""Actions of operators and bonds outside the usual: H without an output where N has one, groups of many
labels, blocks of many elements; what an action reports and what its tuner times.

The bounds are those of the other FP64 parity tests: 1e-10 of the largest entry (the forms differ from the
oracle only in summation order).
"""
import numpy as np
import pytest

from oracle import mpo as M, mps as S
from paper_1703_04789_gb300 import inputs
from tests.gpu_util import masked_random_two_site, require_gpu


def _three_body():
    """T + T^T on four orbitals, T moving three electrons from the right half to the left one: the middle bond
    has channels of charge +3 and -3 only."""
    one, z = np.eye(2), np.diag([1.0, -1.0])
    up = np.array([[0.0, 0.0], [1.0, 0.0]])
    ca, cb = np.kron(up, one), np.kron(z, up)
    pair, par = ca @ cb, np.kron(z, z)
    W = [np.zeros((1, 2, 4, 4)), np.zeros((2, 2, 4, 4)), np.zeros((2, 2, 4, 4)), np.zeros((2, 1, 4, 4))]
    W[0][0, 0], W[0][0, 1] = pair, pair.T
    W[1][0, 0], W[1][1, 1] = ca @ par, par @ ca.T
    W[2][0, 0], W[2][1, 1] = ca.T, ca
    W[3][0, 0], W[3][1, 0] = pair.T, pair
    return W


@pytest.mark.gpu
@pytest.mark.parametrize("opts", [{}, {"fp64_tensor_cores": True}, {"batched": False}])
def test_channels_of_charge_three_only(opts):
    require_gpu()
    from paper_1703_04789_gb300 import Spmps
    K, N, twoM, twoS, D, G = 4, 4, 0, 0, 16, 3
    sites = _three_body()
    labels, tens = inputs.random_mps(K, N, twoM, D, 4)
    P = S.prepare(labels, tens, sites, twoS, twoM, G)
    dev = Spmps(K, N, twoM, twoS, G, D, **opts)
    dev.set_mpo(sites)
    dev.set_mps(P.mps.labels, P.mps.A, center=0)
    P.build_left(K - 2)
    rng = np.random.default_rng(1)
    for k in range(K - 1):
        ql, qr = P.mps.labels[k], P.mps.labels[k + 2]
        lay = dev.x_layout(k)
        x = masked_random_two_site(ql, qr, rng)
        y_ref, z_ref = P.apply(x, k)
        # another vector first: what an output that is not formed would hold
        dev.apply_heff_host(k, rng.standard_normal(lay["n_x"]))
        y, z = dev.apply_heff_host(k, dev.pack(x, lay, ql, qr))
        assert np.abs(dev.unpack(z, lay, ql, qr) - z_ref).max() <= 1e-10 * max(1.0, np.abs(z_ref).max())
        assert np.abs(dev.unpack(y, lay, ql, qr) - y_ref).max() <= 1e-10 * max(1.0, np.abs(y_ref).max())
    dev.close()


@pytest.mark.gpu
@pytest.mark.parametrize("opts", [{}, {"fp64_tensor_cores": True}, {"batched": False}, {"m_screen": 1e-3}])
def test_costs_are_those_of_the_launches(opts):
    """The flops that the costs and the statistics report for an action are those of the kernels it ran."""
    require_gpu()
    import torch
    from paper_1703_04789_gb300 import Spmps
    labels, tens = inputs.random_mps(8, 8, 0, 32, 1)
    dev = Spmps(8, 8, 0, 0, 5, 32, **opts)
    dev.set_hubbard(1.0, 4.0)
    dev.set_mps(labels, tens, center=0)
    x = torch.ones(dev.x_layout(3)["n_x"], dtype=torch.float64, device="cuda")
    y, z = torch.empty_like(x), torch.empty_like(x)
    dev.apply_heff(3, x, y, z)
    costs, bytes_ = dev.apply_costs(3)
    for outs, want in (((y, z), costs.sum()), ((y, None), dev.apply_costs(3)[0][0].sum())):
        before = dev.stats()["apply_flops_total"]
        dev.profile(True)
        dev.apply_heff(3, x, *outs)
        ran = sum(dev.kernel_stats(kind)["flops"] for kind in (0, 1, 8, 9))
        dev.profile(False)
        assert abs(ran - want) <= 1e-12 * want
        assert abs(dev.stats()["apply_flops_total"] - before - ran) <= 1e-12 * dev.stats()["apply_flops_total"]
    assert (costs[1][0] == 0) == (bytes_[1][0] == 0)
    dev.close()


@pytest.mark.gpu
@pytest.mark.parametrize("K,D,G,opts,choice", [
    (8, 32, 5, {}, False),
    (8, 32, 5, {"fp64_tensor_cores": True}, False),    # no tiles
    (16, 200, 5, {}, False),                           # 51 outputs a warp of the chip
    (16, 200, 24, {}, True),                           # 244: 256 and 128 outputs a warp differ
    (16, 200, 24, {"fp64_tensor_cores": True}, False),
])
def test_autotuner_times_only_what_differs(K, D, G, opts, choice):
    """Launches of the first action at a site with and without the autotuner: the same number where no policy
    changes a work list (a launch of up to 128 outputs of phase C per warp that the chip holds; split products)."""
    require_gpu()
    from paper_1703_04789_gb300 import Spmps
    labels, tens = inputs.random_mps(K, K, 0, D, 1)
    launches, z = [], []
    for tuned in (False, True):
        dev = Spmps(K, K, 0, 0, G, D, autotune=tuned, **opts)
        dev.set_hubbard(1.0, 4.0)
        dev.set_mps(labels, tens, center=0)
        x = np.random.default_rng(3).standard_normal(dev.x_layout(K // 2 - 1)["n_x"])
        z.append(dev.apply_heff_host(K // 2 - 1, x)[1])
        launches.append(dev.stats()["launches"])
        dev.close()
    assert (launches[1] > launches[0]) == choice and launches[1] - launches[0] <= 72
    assert np.abs(z[1] - z[0]).max() <= 1e-12 * max(1.0, np.abs(z[0]).max())


def _one_electron_per_site(K, seed):
    """A raw state with one electron on every site and every spin label a bond can have, dimension 1 each: bond i
    has the labels (i, 2m) of one particle number, up to K / 2 + 1 of them."""
    rng = np.random.default_rng(seed)
    half = K // 2
    labels = [np.array([(i, 2 * na - i) for na in range(max(0, half - (K - i)), min(i, half) + 1)], dtype=np.int64)
              for i in range(K + 1)]
    tens = [np.where(S.site_mask(labels[i], labels[i + 1]),
                     rng.uniform(0.5, 1.5, (labels[i].shape[0], 4, labels[i + 1].shape[0])), 0.0) for i in range(K)]
    return labels, tens


@pytest.mark.gpu
@pytest.mark.parametrize("opts", [{}, {"fp64_tensor_cores": True}, {"batched": False}])
def test_groups_of_more_labels_than_mask_bits(opts):
    """67 labels of one particle number: those from the 64th on share a bit, and T1 starts at zero."""
    require_gpu()
    from paper_1703_04789_gb300 import Spmps
    K, G, k = 132, 2, 64
    labels, tens = _one_electron_per_site(K, 5)
    sites = M.hubbard_mpo(K, 1.0, 4.0)
    P = S.prepare(labels, tens, sites, 0, 0, G)
    ql, qr = P.mps.labels[k], P.mps.labels[k + 2]
    assert qr.shape[0] == 67
    dev = Spmps(K, K, 0, 0, G, 80, **opts)
    dev.set_mpo(sites)
    dev.set_mps(P.mps.labels, P.mps.A, center=0)
    P.build_left(k)
    lay = dev.x_layout(k)
    x = masked_random_two_site(ql, qr, np.random.default_rng(1))
    y_ref, z_ref = P.apply(x, k)
    dev.apply_heff_host(k, np.full(lay["n_x"], 1e3))  # what a column that is not written would hold
    y, z = dev.apply_heff_host(k, dev.pack(x, lay, ql, qr))
    assert np.abs(dev.unpack(y, lay, ql, qr) - y_ref).max() <= 1e-10 * np.abs(y_ref).max()
    assert np.abs(dev.unpack(z, lay, ql, qr) - z_ref).max() <= 1e-10 * np.abs(z_ref).max()
    dev.close()


@pytest.mark.gpu
@pytest.mark.parametrize("D,site", [(40, 3), (150, 3), (150, 1)])
def test_separate_combination_over_several_passes(D, site):
    """Active-space operator on eight orbitals: too many inputs for the fused form; at D = 150 the blocks have
    more elements than a CTA takes in one pass (512), at D = 40 fewer."""
    require_gpu()
    from paper_1703_04789_gb300 import Spmps, mpo_from_integrals
    K, N, G = 8, 8, 3
    h1, eri, _ = inputs.synthetic_active_space(K, 7)
    sites = mpo_from_integrals(h1, eri, 0.0)
    labels, tens = inputs.random_mps(K, N, 0, D, 4)
    P = S.prepare(labels, tens, sites, 0, 0, G)
    dev = Spmps(K, N, 0, 0, G, D)
    dev.set_mpo(sites)
    dev.set_mps(P.mps.labels, P.mps.A, center=0)
    P.build_left(site)
    ql, qr = P.mps.labels[site], P.mps.labels[site + 2]
    lay = dev.x_layout(site)
    x = masked_random_two_site(ql, qr, np.random.default_rng(1))
    y_ref, z_ref = P.apply(x, site)
    y, z = dev.apply_heff_host(site, dev.pack(x, lay, ql, qr))
    assert np.abs(dev.unpack(y, lay, ql, qr) - y_ref).max() <= 1e-10 * max(1.0, np.abs(y_ref).max())
    assert np.abs(dev.unpack(z, lay, ql, qr) - z_ref).max() <= 1e-10 * max(1.0, np.abs(z_ref).max())
    dev.close()

"""Order between a caller's stream and the handle's own.

An action on a caller's stream uses the handle's workspaces, environments and work lists and returns before
it has run; everything that the handle does later, on whichever stream, has to wait for it on the device.
A sleep on the caller's stream keeps its action from running, so that the order shows without a race.  Results
are compared for equality: the kernels are deterministic.
"""
import time

import numpy as np
import pytest

from oracle import mpo as M, mps as S
from paper_1703_04789_gb300 import inputs
from tests.gpu_util import require_gpu

CASE = (8, 8, 0, 0, 32, 5, 1, 4.0)
SLEEP = 600_000_000  # clock cycles: 0.3 s at 2 GHz


def _handle(**opts):
    from paper_1703_04789_gb300 import Spmps
    L, N, twoM, twoS, D, G, seed, U = CASE
    labels, tens = inputs.random_mps(L, N, twoM, D, seed)
    P = S.prepare(labels, tens, M.hubbard_mpo(L, 1.0, U), twoS, twoM, G)
    dev = Spmps(L, N, twoM, twoS, G, D, **opts)
    dev.set_hubbard(1.0, U)
    dev.set_mps(P.mps.labels, P.mps.A, center=0)
    return dev


def _vectors(dev, k, seed):
    import torch
    x = torch.tensor(np.random.default_rng(seed).standard_normal(dev.x_layout(k)["n_x"]), device="cuda")
    return x, torch.empty_like(x), torch.empty_like(x)


@pytest.mark.gpu
@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("later", ["own", "side"])
def test_later_work_waits_for_the_action_on_the_callers_stream(noalloc, later):
    require_gpu()
    import torch
    dev = _handle()
    x, y, z = _vectors(dev, 3, 1)
    x2, y2, z2 = _vectors(dev, 3, 2)
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    if later == "own":
        second = torch.cuda.ExternalStream(dev.stream_handle())
    for s in (first, second):  # plan, environments and events
        dev.apply_heff(3, x, y, z, stream=s)
        (dev.apply_heff_noalloc if noalloc else dev.apply_heff)(3, x2, y2, z2, stream=s)
    torch.cuda.synchronize()
    want, want2 = (y.clone(), z.clone()), (y2.clone(), z2.clone())
    torch.cuda.synchronize()
    with torch.cuda.stream(first):
        torch.cuda._sleep(SLEEP)
    (dev.apply_heff_noalloc if noalloc else dev.apply_heff)(3, x, y, z, stream=first)
    dev.apply_heff(3, x2, y2, z2, stream=None if later == "own" else second)
    time.sleep(0.02)
    running, waiting = not first.query(), not second.query()
    torch.cuda.synchronize()
    assert running and waiting
    assert torch.equal(y, want[0]) and torch.equal(z, want[1])
    assert torch.equal(y2, want2[0]) and torch.equal(z2, want2[1])
    dev.close()


@pytest.mark.gpu
@pytest.mark.parametrize("opts", [{}, {"fp64_tensor_cores": True}, {"precision": "3xtf32"}])
def test_calls_on_several_streams_equal_serial_calls(opts):
    """Actions at several sites on three callers' streams and the handle's, environments built in between, the
    last one on a caller's stream, then a step and the energy, which overwrite what it reads."""
    require_gpu()
    import torch

    def calls(streams):
        dev = _handle(**opts)
        out = []
        for i, k in enumerate([0, 5, 3, 3, 6, 1, 5, 3, 0]):
            x, y, z = _vectors(dev, k, 10 + i)
            torch.cuda.current_stream().synchronize()
            s = streams[i % len(streams)]
            if s is not None:
                with torch.cuda.stream(s):
                    torch.cuda._sleep(SLEEP // 50)
            dev.apply_heff(k, x, y, z, stream=s)
            if len(streams) == 1:
                torch.cuda.synchronize()
            out += [x, y, z]
        theta, _ = dev.optimize_step(0, True, allow_not_converged=True)
        energy, norm = dev.energy()
        torch.cuda.synchronize()
        dev.close()
        return [t.cpu().numpy() for t in out], (theta, energy, norm)

    serial, scalars = calls([None])
    got, scalars2 = calls([torch.cuda.Stream(), None, torch.cuda.Stream(), torch.cuda.Stream()])
    assert all(np.array_equal(a, b) for a, b in zip(serial, got))
    assert scalars == scalars2


@pytest.mark.gpu
def test_captured_action_replays():
    """Capture on a caller's stream (relaxed mode: the call waits on the host for the handle's own stream), with an
    earlier action on that stream that the handle has not waited for yet."""
    require_gpu()
    import torch
    dev = _handle()
    x, y, z = _vectors(dev, 3, 1)
    s = torch.cuda.Stream()
    dev.apply_heff(3, x, y, z, stream=s)
    torch.cuda.synchronize()
    want = y.clone(), z.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s, capture_error_mode="relaxed"):
        dev.apply_heff(3, x, y, z, stream=s)
    x2, y2, z2 = _vectors(dev, 3, 2)
    torch.cuda.synchronize()
    dev.apply_heff(3, x2, y2, z2)
    y.zero_(), z.zero_()
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, want[0]) and torch.equal(z, want[1])
    dev.close()

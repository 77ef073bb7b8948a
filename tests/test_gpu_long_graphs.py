"""Graphs of several intervals: captured behind queued work, so that no call
waits for them, and with the states and samples of single intervals."""
import time

import numpy as np
import pytest
import torch

import spin_inputs

pytestmark = pytest.mark.gpu

KW = dict(J=1.0, D=0.05, H=(0.01, -0.02, 0.02), lam=0.05, T=1.0, dt=0.05, seed=3)


def test_no_call_waits_for_a_capture(gpu):
    """Ten calls of ten intervals on fresh handles, M and E read after each: from
    the second call on (the first captures the interval itself) none takes much
    longer than the fastest.  Capturing the longer graphs in front of the work
    made one of them 1.8 times as long; 1.4 for noise."""
    p = gpu.Params(32, 32, 32, R=1, **KW)
    s0 = torch.from_numpy(spin_inputs.random_spins(32, 32, 32, seed=2)).cuda()
    best = np.full(10, np.inf)
    for _ in range(9):
        lat = gpu.Lattice(p, s0)
        torch.cuda.synchronize()
        for k in range(10):
            t = time.perf_counter()
            lat.step(10)
            lat.observables()
            best[k] = min(best[k], time.perf_counter() - t)
        lat.close()
    assert best[1:].max() < 1.4 * best[1:].min(), best


# calls of many lengths, so that graphs of every length are captured in the
# middle and at the end of calls and begin in either buffer (an odd number of
# steps without noise changes it), against one step per call
@pytest.mark.parametrize("R,noise", [(1, 1), (1, 0), (2, 1), (3, 0), (5, 1)])
def test_calls_of_many_lengths(gpu, R, noise):
    p = gpu.Params(11, 10, 9, R=R, noise=noise, **KW)
    s0 = torch.from_numpy(spin_inputs.random_spins(11, 10, 9, seed=2))
    a, b = gpu.Lattice(p, s0), gpu.Lattice(p, s0)
    n = 0
    for c in (1, 9, 2, 2, 10, 4, 7, 23, 3, 16, 8, 8, 31, 5, 40, 1, 6):
        a.step(c * R)
        n += c * R
        if c == 7:
            a.step(R + 1)     # then begins inside an interval
            a.step(R - 1)
            n += 2 * R
    for _ in range(n):
        b.step(1)
    torch.cuda.synchronize()
    assert a.n == b.n == n and torch.equal(a.state, b.state)
    assert a.samples() == b.samples()

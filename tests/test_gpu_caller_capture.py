"""Calls on a stream that the caller captures: the graph has ordinary edges
only, and replaying it does what the calls do."""
import numpy as np
import pytest
import torch

import spin_inputs
from graph_capture import Captured

pytestmark = pytest.mark.gpu

SHAPE = (20, 18, 12)
KW = dict(J=0.9, D=0.15, H=(0.05, -0.1, 0.2), lam=0.1, T=0.7, dt=0.07, seed=77)


def spins(shape, dtype=torch.float32):
    return torch.from_numpy(spin_inputs.random_spins(*shape, seed=3)).to(dtype)


# an interval captured before the handle has replayed one of its own and after
@pytest.mark.parametrize("before", [0, 3])
@pytest.mark.parametrize("integ,precision,R,shape", [
    ("RK4", 32, 2, SHAPE), ("RK4", 32, 3, SHAPE), ("RK4", 64, 2, SHAPE), ("HEUN", 32, 1, (90, 68, 66)),
    ("RK5_BUTCHER", 32, 2, SHAPE), ("RK4", 64, 3, (30, 27, 26))])
def test_steps(gpu, integ, precision, R, shape, before):
    p = gpu.Params(*shape, R=R, precision=precision, integrator=getattr(gpu, integ), **KW)
    st = torch.cuda.Stream()
    lat = gpu.Lattice(p, spins(shape), stream=st)
    torch.cuda.synchronize()
    lat.step(before * R)
    g = Captured(st, lambda: lat.step(R))
    assert g.plain_edges()
    g.replay(4)
    ref = gpu.Lattice(p, spins(shape)).step((before + 4) * R)
    torch.cuda.synchronize()
    assert torch.equal(lat.state, ref.state)
    assert lat.samples() == ref.samples()
    g.close()


def test_batch_steps(gpu):
    L, R = [12, 9], 2
    p = gpu.Params(1, 1, 1, R=R, **{k: v for k, v in KW.items() if k != "T"})
    s0 = [spin_inputs.random_spins(v, v, v, seed=v).astype(np.float32) for v in L]
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    b = gpu.Batch(p, L, [0.7, 0.5], s0, chunk_planes=gpu.batch.DEFAULT_TILING, stream=st)
    torch.cuda.synchronize()
    b.step(2 * R)
    g = Captured(st, lambda: b.step(R))
    assert g.plain_edges()
    g.replay(3)
    ref = gpu.Batch(p, L, [0.7, 0.5], s0, chunk_planes=gpu.batch.DEFAULT_TILING)
    ref.step(5 * R)
    torch.cuda.synchronize()
    for r in range(2):
        assert torch.equal(b.replica_state(r), ref.replica_state(r))
    g.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_observables_noalloc(gpu, dtype):
    st = torch.cuda.Stream()
    s = spins(SHAPE, dtype).cuda()
    out, ref = (torch.zeros(5, dtype=torch.float64, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    call = lambda o, stream: gpu.spin_observables_noalloc(s, 0.8, 0.3, (0.1, -0.2, 0.4), o, bc=1, stream=stream)
    call(ref, st)
    g = Captured(st, lambda: call(out, st))
    assert g.plain_edges()
    for k in range(2):
        s.mul_(-1 if k else 1)
        call(ref, torch.cuda.current_stream())
        torch.cuda.synchronize()
        g.replay()
        assert torch.equal(out, ref)
    g.close()


@pytest.mark.parametrize("precision", [32, 64])
def test_metropolis(gpu, precision):
    p = gpu.Params(*SHAPE, J=1.0, D=0.1, H=(0.0, 0.1, 0.2), T=0.8, precision=precision)
    st = torch.cuda.Stream()
    a, b = spins(SHAPE, p.dtype).cuda(), spins(SHAPE, p.dtype).cuda()
    na, nb = (torch.zeros(1, dtype=torch.int64, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    call = lambda s, n, stream: gpu.spin_metropolis_sweeps(p, s, mc_seed=5, sweep0=2, nsweeps=3, accepted=n, stream=stream)
    g = Captured(st, lambda: call(a, na, st))
    assert g.kernels() == 6 and g.plain_edges()
    g.replay(2)
    for _ in range(2):
        call(b, nb, None)
    torch.cuda.synchronize()
    assert torch.equal(a, b) and torch.equal(na, nb)
    g.close()

"""Rectangular noise with several lanes per replica: the sizes at which the
number of lanes changes."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def spins(gpu, nrep, integ, R, prec):
    p = gpu.Params(1, 1, 1, J=0.0, D=0.4, H=(0.3, -0.2, 0.4), lam=0.2, T=0.0, dt=0.1, R=R, integrator=integ, noise=2,
                   seed=21, precision=prec)
    T = np.linspace(0.05, 1.0, nrep)
    v = np.random.default_rng(4).normal(size=(3, nrep))
    s0 = v / np.linalg.norm(v, axis=0)
    if prec == 32:
        s0 = s0.astype(np.float32).astype(np.float64)
    return T, s0, gpu.SingleSpins(p, T, torch.from_numpy(s0))


# 8, 4, 2 and 1 lanes: the last and the first replica count of each, against the
# oracle on sampled replicas (tolerances of test_gpu_single.py)
@pytest.mark.parametrize("prec,tol", [(64, 1e-12), (32, 2e-5)])
@pytest.mark.parametrize("nrep", [2432, 2433, 4864, 4865, 9728, 9729])
def test_lane_limits(gpu, orc, prec, tol, nrep):
    T, s0, ss = spins(gpu, nrep, 3, 2, prec)
    ss.run(9, average=True).run(12, average=True)
    torch.cuda.synchronize()
    got = ss.state.double().cpu().numpy()
    assert (ss.sz_count.cpu().numpy() == 10).all()
    for r in (0, 1, nrep // 2, nrep - 1):
        q = orc.Params(1, 1, 1, J=0.0, D=0.4, H=(0.3, -0.2, 0.4), lam=0.2, T=float(T[r]), dt=0.1, R=2, integrator=3,
                       seed=21, replica=r)
        ref, _ = orc.run(q, s0[:, r].reshape(3, 1, 1, 1), 21, noise=2)
        assert np.max(np.abs(got[:, r] - ref.reshape(3))) < tol


def test_lanes_do_not_crowd_the_fp64_pipe(gpu):
    """Every lane repeats its replica's steps, so a second warp per scheduler
    would double an FP64 run (R = 40: almost all of it steps).  More replicas than
    the lanes are made for, one lane each, take the time of one warp per
    scheduler and bound the smaller runs; 1.25 for noise of the timing."""
    def us(nrep):
        ss = spins(gpu, nrep, 1, 40, 64)[2]
        ss.run(120)
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            ss.run(120)
            b.record()
            torch.cuda.synchronize()
            best = min(best, 1e3 * a.elapsed_time(b))
        return best

    ref = us(12288)
    for nrep in (2432, 3000, 6144, 9728, 10240):
        assert us(nrep) < 1.25 * ref, nrep

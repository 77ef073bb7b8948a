"""Kernels that start before the kernel before them has finished (pdl.cuh):
what they read has to be what that order of launches gives."""
import numpy as np
import pytest
import torch

import spin_inputs
from gpu_helpers import as_input, orc_params, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


# free spins, a pulse every step or every second one, whole intervals first one
# by one, then from graphs of one and of several: every pulse is drawn with its
# own number (one taken for another would be off by sigma |G| ~ 0.1).  Per pulse
# the angle carries about four roundings of G and the rotation about ten; |G| < 6.
@pytest.mark.parametrize("R", [1, 2])
@pytest.mark.parametrize("shape", [(20, 17, 9), (66, 65, 64)])
def test_every_pulse_has_its_number(gpu, orc, shape, R):
    sigma, n = 0.05, 40
    p = gpu.Params(*shape, J=0.0, D=0.0, H=(0.0, 0.0, 0.0), lam=0.5 / R, T=sigma ** 2, dt=1.0, R=R, seed=5)
    s0 = spin_inputs.random_spins(*shape, seed=3)
    got, lat = run_gpu(gpu, p, s0, n)
    ref, _ = run_oracle(orc, p, s0, n)
    assert np.max(np.abs(got - ref)) < n // R * (4 * 6 * sigma + 10) * 2.0 ** -24
    assert [int(r[0]) for r in lat.samples()] == list(range(R, n + 1, R))


def test_every_batch_pulse_has_its_number(gpu, orc):
    sigma, n, L = 0.05, 24, [8, 19]
    p = gpu.Params(1, 1, 1, J=0.0, D=0.0, H=(0.0, 0.0, 0.0), lam=0.5, dt=1.0, R=1, seed=5)
    s0 = [spin_inputs.random_spins(v, v, v, seed=v).astype(np.float32) for v in L]
    b = gpu.Batch(p, L, [sigma ** 2] * 2, s0, chunk_planes=gpu.batch.DEFAULT_TILING)
    b.step(n)
    torch.cuda.synchronize()
    for r, v in enumerate(L):
        q = gpu.Params(v, v, v, J=0.0, D=0.0, H=(0.0, 0.0, 0.0), lam=0.5, T=sigma ** 2, dt=1.0, R=1, seed=5, replica=r)
        ref, _ = orc.run(orc_params(orc, q), as_input(q, s0[r]), n)
        d = b.replica_state(r).double().cpu().numpy().reshape(3, v, v, v) - ref
        assert np.max(np.abs(d)) < n * (4 * 6 * sigma + 10) * 2.0 ** -24

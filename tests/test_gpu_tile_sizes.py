"""The fused FP32 tile on lattices that take it by themselves, just above the
sizes of the stage kernels (48^3 sites for RK4, 56^3 with site fields, 64^3 and
72^3 for two stages, 96^3 for steps that store their stages)."""
import numpy as np
import pytest
import torch

import spin_inputs
from gpu_helpers import as_input, orc_params, run_gpu, run_oracle

pytestmark = pytest.mark.gpu

KW = dict(J=0.9, D=0.15, H=(0.05, -0.1, 0.2), lam=0.1, T=0.7, dt=0.07, seed=77)


# ragged and flat lattices, both boundaries and equations, with and without site
# fields, against the oracle (one step agrees to 2e-6, three run)
@pytest.mark.parametrize("integ,shape,precession,hsite,bc", [
    ("RK4", (61, 43, 47), 1, False, 1), ("RK4", (200, 201, 3), 0, False, 0),
    ("RK4", (71, 50, 53), 0, True, 1), ("RK4", (300, 301, 2), 1, True, 0),
    ("RK2_MIDPOINT", (87, 61, 53), 0, False, 1), ("HEUN", (301, 291, 3), 1, False, 0),
    ("RK2_MIDPOINT", (91, 67, 63), 1, True, 1), ("HEUN", (401, 331, 3), 0, True, 0)])
def test_tile_against_oracle(gpu, orc, integ, shape, precession, hsite, bc):
    p = gpu.Params(*shape, R=3, integrator=getattr(gpu, integ), precession=precession, bc=bc, **KW)
    s0 = spin_inputs.random_spins(*shape, seed=3)
    hs = spin_inputs.site_fields(*shape, 0.1, seed=4) if hsite else None
    got, _ = run_gpu(gpu, p, s0, 3, h_site=hs)
    ref, _ = run_oracle(orc, p, s0, 3, h_site=hs)
    assert np.max(np.abs(got - ref)) < 3 * 2e-6


# recomputing steps of the adjoint that store their stages in the tile: gradients
# bitwise the same for every K, and the oracle's (bounds of test_gpu_adjoint.py)
@pytest.mark.parametrize("integ,shape,precession,bc,hsite", [
    ("RK4", (97, 95, 97), 1, 0, True), ("RK2_MIDPOINT", (301, 491, 6), 0, 1, False)])
def test_stored_stages_above_the_limit(gpu, orc, integ, shape, precession, bc, hsite):
    p = gpu.Params(*shape, R=3, integrator=getattr(gpu, integ), precession=precession, bc=bc, **KW)
    s0 = spin_inputs.random_spins(*shape, seed=11)
    hs = spin_inputs.site_fields(*shape, 0.1, seed=13) if hsite else None

    def grad(K):
        lat = gpu.Lattice(p, torch.from_numpy(s0), h_site=None if hs is None else torch.from_numpy(hs))
        lat.record(K, 3)
        lat.step(3)
        g = lat.backward([0.3, -0.2, 0.7], 1.0, field_grad=True, state_grad=True)
        return [np.array([g["J"]]), np.array([g["D"]]), np.array(g["H"]), g["h"].cpu().numpy(),
                g["s0"].double().cpu().numpy()]

    got = grad(2)
    for K in (1, 3):
        assert all(np.array_equal(a, b) for a, b in zip(got, grad(K)))
    ref = orc.adjoint(orc_params(orc, p), as_input(p, s0), 3, [0.3, -0.2, 0.7], 1.0,
                      h_site=None if hs is None else as_input(p, hs))
    for g, r in zip(got, (ref["J"], ref["D"], ref["H"], ref["h"], ref["s0"])):
        r = np.asarray(r, float).ravel()
        assert np.max(np.abs(g.ravel() - r)) < 1e-5 * np.max(np.abs(r))


# odd intervals, whose pulse goes back to the buffer the interval began in:
# single steps, whole intervals (eager, then graphs) and recorded runs, bitwise;
# the last lattices lie above 2^20 sites, where graphs hold one interval and
# ordinary edges
@pytest.mark.parametrize("integ,shape,R", [
    ("RK4", (61, 43, 47), 1), ("RK4", (61, 43, 47), 3), ("HEUN", (87, 61, 53), 3), ("RK4", (103, 101, 102), 3),
    ("RK5_BUTCHER", (103, 101, 102), 1), ("RK4", (256, 257, 17), 5)])
def test_odd_intervals_of_the_tile(gpu, integ, shape, R):
    p = gpu.Params(*shape, R=R, integrator=getattr(gpu, integ), **KW)
    s0 = torch.from_numpy(spin_inputs.random_spins(*shape, seed=3))
    one, whole, rec = (gpu.Lattice(p, s0) for _ in range(3))
    n = 4 * R + 2
    for _ in range(n):
        one.step(1)
    whole.step(n)
    rec.record(R, n)
    rec.step(n)
    torch.cuda.synchronize()
    assert torch.equal(one.state, whole.state) and torch.equal(one.state, rec.state)
    assert one.samples() == whole.samples() == rec.samples()

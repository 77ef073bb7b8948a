"""SPIN_TMA=1 and SPIN_TMEM=1 choose the fused tile at every size, small
lattices (otherwise one kernel per stage) among them; the states are bitwise the
same either way."""
import numpy as np
import pytest
import torch

import spin_inputs
from graph_capture import Captured

pytestmark = pytest.mark.gpu

KW = dict(J=0.9, D=0.15, H=(0.05, -0.1, 0.2), lam=0.1, T=0.7, dt=0.07, R=3, seed=77)


@pytest.fixture
def no_switches(monkeypatch):
    for v in ("SPIN_TMA", "SPIN_TMEM"):
        monkeypatch.delenv(v, raising=False)
    return monkeypatch


@pytest.mark.parametrize("switch", [None, "SPIN_TMA", "SPIN_TMEM"])
@pytest.mark.parametrize("integ,hsite,stages", [("RK4", False, 4), ("RK4", True, 4), ("HEUN", False, 2)])
def test_kernels_of_a_small_step(gpu, no_switches, switch, integ, hsite, stages):
    """A step without pulse or sample: one kernel where a switch is set, one per
    stage where none is."""
    shape = (24, 20, 8)
    st = torch.cuda.Stream()
    hs = torch.from_numpy(spin_inputs.site_fields(*shape, 0.1, seed=4)) if hsite else None
    lat = gpu.Lattice(gpu.Params(*shape, integrator=getattr(gpu, integ), **{**KW, "R": 9}),
                      torch.from_numpy(spin_inputs.random_spins(*shape, seed=3)), h_site=hs, stream=st)
    torch.cuda.synchronize()
    if switch:
        no_switches.setenv(switch, "1")
    g = Captured(st, lambda: lat.step(1))
    assert g.kernels() == (1 if switch else stages)
    g.close()


# the tile at its edges (ragged, narrow and thin lattices, one plane, both
# boundaries, both equations, site fields) against the stage kernels, whose
# neighbours are plain indices; RK4 lattices with sides that are multiples of 4
# stage their planes by tensor-map copies with SPIN_TMA=1
# (with SPIN_TMEM=1 in the tensor-memory step)
@pytest.mark.parametrize("switch,integ,hsite", [("SPIN_TMEM", "RK4", False)] + [
    ("SPIN_TMA", i, h) for i in ("RK4", "RK2_MIDPOINT", "HEUN") for h in (False, True)])
@pytest.mark.parametrize("shape,precession,bc", [
    ((37, 21, 13), 1, 0), ((45, 37, 27), 0, 1), ((2, 3, 5), 1, 1), ((1, 1, 1), 0, 0), ((129, 151, 1), 1, 1),
    ((1, 1, 700), 1, 0), ((7, 90, 3), 0, 0), ((28, 20, 11), 1, 1), ((64, 36, 17), 0, 0), ((24, 16, 9), 1, 0)])
def test_tile_equals_stages(gpu, no_switches, switch, integ, shape, precession, bc, hsite):
    p = gpu.Params(*shape, integrator=getattr(gpu, integ), precession=precession, bc=bc, **KW)
    s0 = torch.from_numpy(spin_inputs.random_spins(*shape, seed=3))
    hs = torch.from_numpy(spin_inputs.site_fields(*shape, 0.1, seed=4)) if hsite else None
    a = gpu.Lattice(p, s0, h_site=hs).step(13)
    no_switches.setenv(switch, "1")
    b = gpu.Lattice(p, s0, h_site=hs).step(13)
    torch.cuda.synchronize()
    assert torch.equal(a.state, b.state) and a.samples() == b.samples()


# recomputing steps that store their stages (k_step_patch_store)
@pytest.mark.parametrize("integ", ["RK4", "RK2_MIDPOINT"])
@pytest.mark.parametrize("shape,precession,bc,hsite", [((37, 21, 13), 1, 0, False), ((33, 9, 3), 0, 1, True),
                                                       ((45, 37, 27), 1, 1, True), ((2, 3, 5), 0, 0, False)])
def test_stored_stages_of_tile_and_stage_kernels(gpu, no_switches, integ, shape, precession, bc, hsite):
    p = gpu.Params(*shape, integrator=getattr(gpu, integ), precession=precession, bc=bc, **KW)
    s0 = torch.from_numpy(spin_inputs.random_spins(*shape, seed=3))
    hs = torch.from_numpy(spin_inputs.site_fields(*shape, 0.1, seed=4)) if hsite else None

    def grad():
        lat = gpu.Lattice(p, s0, h_site=hs)
        lat.record(3, 7)
        lat.step(7)
        g = lat.backward([0.3, -0.2, 0.7], 1.0, field_grad=True, state_grad=True)
        return np.concatenate([[g["J"], g["D"]], g["H"], g["h"].cpu().numpy().ravel(), g["s0"].cpu().numpy().ravel()])

    a = grad()
    no_switches.setenv("SPIN_TMA", "1")
    assert np.array_equal(a, grad())

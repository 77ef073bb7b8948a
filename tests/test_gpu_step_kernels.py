"""The step kernels at the sizes where their geometry can go wrong, against
the FP64 oracle on the same inputs and noise (tolerances of the parity tests:
one step agrees to 1e-13 in FP64 and 2e-6 in FP32, three steps run here)."""
import numpy as np
import pytest

import spin_inputs
from gpu_helpers import run_gpu, run_oracle

pytestmark = pytest.mark.gpu


def _compare(gpu, orc, shape, tol, hsite=False, **kw):
    nx, ny, nz = shape
    p = gpu.Params(nx, ny, nz, J=0.9, D=0.15, H=(0.05, -0.1, 0.2), lam=0.1, T=0.7, dt=0.07, R=3, seed=77, replica=2,
                   **kw)
    s0 = spin_inputs.random_spins(nx, ny, nz, seed=3)
    hs = spin_inputs.site_fields(nx, ny, nz, 0.1, seed=4) if hsite else None
    got, _ = run_gpu(gpu, p, s0, 3, h_site=hs)
    ref, _ = run_oracle(orc, p, s0, 3, h_site=hs)
    assert np.max(np.abs(got - ref)) < tol


# one-warp blocks up to 19456 sites, four-warp blocks beyond; a last block of
# one site, of one site less than full; sides of 1 and 2 (neighbours coincide)
@pytest.mark.parametrize("integ", ["RK4", "RK2_MIDPOINT", "HEUN"])
@pytest.mark.parametrize("shape,precession,hsite,bc", [
    ((32, 32, 19), 1, False, 0),
    ((29, 11, 61), 1, True, 1),
    ((31, 1, 1), 0, False, 1),
    ((1, 2, 97), 1, True, 0),
    ((3, 43, 152), 0, False, 0),
])
def test_fp64_stage_kernels(gpu, orc, integ, shape, precession, hsite, bc):
    _compare(gpu, orc, shape, 1e-13, hsite=hsite, precision=64, integrator=getattr(gpu, integ),
             precession=precession, bc=bc)

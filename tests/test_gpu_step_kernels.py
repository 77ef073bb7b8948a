"""The step kernels at the sizes where their geometry can go wrong, against
the FP64 oracle on the same inputs and noise (tolerances of the parity tests:
one step agrees to 1e-13 in FP64 and 2e-6 in FP32, three steps run here)."""
import numpy as np
import pytest
import torch

import spin_inputs
from gpu_helpers import as_input, orc_params, run_gpu, run_oracle

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


# four lanes per site up to 10944 sites: a last block of one site, exactly the
# line, one site beyond it; sides of 1, free faces, site fields
@pytest.mark.parametrize("integ", ["RK4", "RK2_MIDPOINT", "HEUN"])
@pytest.mark.parametrize("shape,precession,hsite,bc", [
    ((1, 1, 1), 1, True, 0), ((3, 11, 1), 0, False, 1), ((5, 5, 5), 1, False, 1),
    ((16, 18, 38), 1, True, 1), ((5, 11, 199), 0, True, 0)])
def test_fp64_component_lanes(gpu, orc, integ, shape, precession, hsite, bc):
    _compare(gpu, orc, shape, 1e-13, hsite=hsite, precision=64, integrator=getattr(gpu, integ),
             precession=precession, bc=bc)


# the last FP64 stage without renormalisation (its result scaled back), and
# spins of 1e-30, whose squared length lies outside the range of the short
# reciprocal root; four lanes, one thread per site, and the integer sums
@pytest.mark.parametrize("integ,precession", [("RK4", 1), ("RK2_MIDPOINT", 0)])
@pytest.mark.parametrize("shape", [(7, 6, 5), (23, 22, 24), (28, 27, 26)])
@pytest.mark.parametrize("renorm,scale", [(0, 1.0), (1, 1e-30)])
def test_fp64_last_stage_forms(gpu, orc, integ, precession, shape, renorm, scale):
    p = gpu.Params(*shape, J=0.9, D=0.15, H=(0.05, -0.1, 0.2), lam=0.1, T=0.7, dt=0.07, R=3, seed=77, replica=2,
                   precision=64, renorm=renorm, integrator=getattr(gpu, integ), precession=precession)
    s0 = scale * spin_inputs.random_spins(*shape, seed=3)
    got, _ = run_gpu(gpu, p, s0, 3)
    ref, _ = run_oracle(orc, p, s0, 3)
    assert np.max(np.abs(got - ref)) < 1e-13


# free spins (J = D = H = 0): three pulses with sigma at both sides of the
# series limit 0.35, far above it (general form), and angles from ~0 to beyond
# phi^2 = 4.  Per pulse the angle carries about four roundings of G, relative,
# so phi times that, and the rotation about ten more; |G| < 6 here.
@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("sigma", [0.01, 0.3499, 0.3501, 1.55])
def test_pulse_rotation_forms(gpu, orc, prec, sigma):
    n = (33, 17, 40)
    p = gpu.Params(*n, J=0.0, D=0.0, H=(0.0, 0.0, 0.0), lam=0.5, T=sigma ** 2, dt=1.0, R=1, seed=5, precision=prec)
    s0 = spin_inputs.random_spins(*n, seed=3)
    got, _ = run_gpu(gpu, p, s0, 3)
    ref, _ = run_oracle(orc, p, s0, 3)
    tol = 1e-13 if prec == 64 else 3 * (4 * 6 * sigma + 10) * 2.0 ** -24
    assert np.max(np.abs(got - ref)) < tol


def test_noise_uniforms_small_words(gpu):
    """2^22 draws, so that words below 2^44 (the conversion's other branch, one
    in 2^20) occur: Gaussians against numpy's from the same words, whose
    uniforms the FP32 path rounds once to float."""
    words, g32 = gpu.spin_noise_draw(9, 3, 1, 1 << 22, precision=32)
    torch.cuda.synchronize()
    w = words.cpu().numpy().view(np.uint64)
    assert int((w < np.uint64(1 << 44)).sum()) > 0
    u = (((w >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53).astype(np.float32).astype(np.float64)
    r0, r2 = np.sqrt(-2 * np.log(u[:, 0])), np.sqrt(-2 * np.log(u[:, 2]))
    a, b = 2 * np.pi * u[:, 1], 2 * np.pi * u[:, 3]
    ref = np.stack([r0 * np.cos(a), r0 * np.sin(a), r2 * np.cos(b)], 1)
    assert np.max(np.abs(g32.cpu().numpy() - ref)) < 1e-5


# rows fewer than, equal to and beyond one block's warps and the grid; row ends
# inside and at a lane's stride; M and E against a plain FP64 reduction (FP32
# terms: bounds of the parity tests)
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("shape", [(1, 1, 1), (33, 1, 1), (1, 1, 17), (32, 4, 4), (31, 5, 3), (70, 16, 305)])
def test_observables_reduction(gpu, dtype, bc, shape):
    nx, ny, nz = shape
    s = torch.from_numpy(spin_inputs.random_spins(nx, ny, nz, seed=6)).to("cuda", dtype)
    h = torch.from_numpy(spin_inputs.site_fields(nx, ny, nz, 0.3, seed=7)).to("cuda", dtype)
    J, D, H = 0.8, 0.3, (0.1, -0.2, 0.4)
    out = torch.zeros(5, dtype=torch.float64, device="cuda")
    gpu.spin_observables_noalloc(s, J, D, H, out, h_site=h, bc=bc)
    x, f = s.double(), h.double() + torch.tensor(H, dtype=torch.float64, device="cuda").reshape(3, 1, 1, 1)
    bonds = x.new_zeros(())
    for d in (1, 2, 3):
        p = x * torch.roll(x, -1, d)
        bonds = bonds + (p.narrow(d, 0, x.shape[d] - 1).sum() if bc else p.sum())
    n = nx * ny * nz
    E = float((-J * bonds - D * x[2].square().sum() - (f * x).sum()) / n)
    M = (x.reshape(3, -1).sum(1) / n).tolist()
    got = out.tolist()
    tm, te = (1e-6, 5e-6) if dtype == torch.float32 else (1e-13, 1e-13)
    assert max(abs(a - b) for a, b in zip(got[:3], M)) < tm and abs(got[3] - E) < te and got[4] == 0
    s[1, nz // 2, ny // 2, nx - 1] = float("inf")
    s[0, 0, 0, 0] = float("nan")
    gpu.spin_observables_noalloc(s, J, D, H, out, h_site=h, bc=bc)
    assert out[4].item() == (1 if n == 1 else 2 if (nz // 2, ny // 2, nx - 1) != (0, 0, 0) else 1)


# odd intervals: the pulse goes back to the buffer the interval began in; whole
# intervals (eager, then graphs), single steps and recorded runs end in the same
# states, samples and checkpoints, bit for bit
@pytest.mark.parametrize("integ", ["RK4", "RK2_MIDPOINT", "RK5_BUTCHER"])
@pytest.mark.parametrize("R", [1, 3, 5])
def test_odd_intervals_bitwise(gpu, integ, R):
    p = gpu.Params(30, 17, 12, J=0.9, D=0.15, H=(0.05, -0.1, 0.2), lam=0.1, T=0.7, dt=0.07, R=R, seed=7,
                   integrator=getattr(gpu, integ))
    s0 = torch.from_numpy(spin_inputs.random_spins(30, 17, 12, seed=3))
    one, whole, rec = (gpu.Lattice(p, s0) for _ in range(3))
    n = 4 * R + 2
    states = [one.state.clone()]
    for _ in range(n):
        one.step(1)
        states.append(one.state.clone())
    whole.step(n)
    rec.record(R, n)
    rec.step(n)
    assert torch.equal(one.state, whole.state) and torch.equal(one.state, rec.state)
    assert one.samples() == whole.samples() == rec.samples()
    slots = rec.store.view(torch.float32)[: (n // R + 1) * one.state.numel()].reshape(n // R + 1, -1)
    for c in range(n // R + 1):
        assert torch.equal(slots[c], states[c * R].reshape(-1)), c


# the pair kernel (from 65536 replicas; an odd count leaves one replica alone),
# the axial right-hand side (H along z, with anisotropy) and calls that end
# mid-interval, against the oracle on sampled replicas (tolerances of
# test_gpu_single.py)
@pytest.mark.parametrize("integ,precession", [(0, 1), (1, 1), (1, 0), (3, 1)])
@pytest.mark.parametrize("H", [(0.0, 0.0, 0.9), (0.3, -0.2, 0.4)])
@pytest.mark.parametrize("nrep", [131, 98305])
def test_single_pairs(gpu, orc, integ, precession, H, nrep):
    p = gpu.Params(1, 1, 1, J=0.0, D=0.4, H=H, lam=0.2, T=0.0, dt=0.1, R=6, integrator=integ, precession=precession,
                   seed=21, precision=32)
    T = np.linspace(0.05, 1.0, nrep)
    v = np.random.default_rng(4).normal(size=(3, nrep))
    s0 = (v / np.linalg.norm(v, axis=0)).astype(np.float32)
    ss = gpu.SingleSpins(p, T, torch.from_numpy(s0))
    ss.run(16, average=True).run(20, average=True)
    torch.cuda.synchronize()
    got, sums = ss.state.double().cpu().numpy(), ss.sz_sum.cpu().numpy()
    assert (ss.sz_count.cpu().numpy() == 6).all()
    for r in (0, 1, 64, nrep // 2 - 1, nrep // 2, nrep // 2 + 1, nrep - 1):
        q = orc.Params(1, 1, 1, J=0.0, D=0.4, H=H, lam=0.2, T=float(T[r]), dt=0.1, R=6, integrator=integ,
                       precession=precession, seed=21, replica=r)
        ref, smp = orc.run(q, s0[:, r].astype(np.float64).reshape(3, 1, 1, 1), 36)
        assert np.max(np.abs(got[:, r] - ref.reshape(3))) < 2e-5
        assert abs(sums[r] - smp[:, 3].sum()) < 6 * 2e-5


def test_noise_fp64_draw(gpu):
    """2^20 FP64 draws (every interval of the logarithm's and the angles'
    tables, uniforms down to 2^-20 and up to 1 - 2^-20) against numpy from the
    same words; 2e-14 as in the parity test: a few roundings of r <= 8.7 here and
    in numpy's argument 2 pi u."""
    words, g = gpu.spin_noise_draw(11, 5, 2, 1 << 20, precision=64)
    torch.cuda.synchronize()
    w = words.cpu().numpy().view(np.uint64)
    u = ((w >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53
    r0, r2 = np.sqrt(-2 * np.log(u[:, 0])), np.sqrt(-2 * np.log(u[:, 2]))
    a, b = 2 * np.pi * u[:, 1], 2 * np.pi * u[:, 3]
    ref = np.stack([r0 * np.cos(a), r0 * np.sin(a), r2 * np.cos(b)], 1)
    assert np.max(np.abs(g.cpu().numpy() - ref)) < 2e-14


# the fixed-point sums of the FP64 stages (beyond 19456 sites): mixed magnitudes
# (components from 1 down to 2^-70), exact zeros, and a non-finite spin, which
# has to reach its neighbours and nobody else
def test_fp64_stage_sums(gpu, orc):
    n = (28, 27, 26)
    g = np.random.default_rng(8)
    s0 = spin_inputs.random_spins(*n, seed=3)
    s0[0] *= 2.0 ** -g.integers(0, 70, s0[0].shape)
    s0[1, :9] = 0.0
    s0[:, 20:] = np.array([0.0, 0.0, 1.0]).reshape(3, 1, 1, 1)
    for J, H in ((1.0, (0.0, 0.0, 0.2)), (0.9, (0.05, -0.1, 0.2))):
        p = gpu.Params(*n, J=J, D=0.15, H=H, lam=0.1, T=0.7, dt=0.07, R=3, seed=77, precision=64)
        got, lat = run_gpu(gpu, p, s0, 3)
        ref, _ = run_oracle(orc, p, s0, 3)
        assert np.max(np.abs(got - ref)) < 1e-13
    bad = torch.from_numpy(s0.copy())
    bad[0, 13, 13, 13] = float("inf")
    p.noise, p.integrator = 0, gpu.RK2_MIDPOINT
    lat = gpu.Lattice(p, bad).step(1)
    z, y, x = torch.where(~torch.isfinite(lat.state).all(0))
    d = (z - 13).abs() + (y - 13).abs() + (x - 13).abs()
    assert int(d.max()) == 2 and len(d) == 25   # two stages: the octahedron of radius 2


# rectangular noise with 8, 4, 2 and 1 lanes per replica (the last warp partly
# idle), calls that end mid-interval, against the oracle on sampled replicas
@pytest.mark.parametrize("prec,tol", [(64, 1e-12), (32, 2e-5)])
@pytest.mark.parametrize("nrep", [3, 2049, 6145, 10241])
@pytest.mark.parametrize("integ,R", [(3, 1), (1, 4)])
def test_single_rect_lanes(gpu, orc, prec, tol, nrep, integ, R):
    p = gpu.Params(1, 1, 1, J=0.0, D=0.4, H=(0.3, -0.2, 0.4), lam=0.2, T=0.0, dt=0.1, R=R, integrator=integ, noise=2,
                   seed=21, precision=prec)
    T = np.linspace(0.05, 1.0, nrep)
    v = np.random.default_rng(4).normal(size=(3, nrep))
    s0 = v / np.linalg.norm(v, axis=0)
    if prec == 32:
        s0 = s0.astype(np.float32).astype(np.float64)
    ss = gpu.SingleSpins(p, T, torch.from_numpy(s0))
    ss.run(10, average=True).run(11, average=True)
    torch.cuda.synchronize()
    got, sums = ss.state.double().cpu().numpy(), ss.sz_sum.cpu().numpy()
    assert (ss.sz_count.cpu().numpy() == 21 // R).all()
    for r in (0, 1, nrep // 2, nrep - 1):
        q = orc.Params(1, 1, 1, J=0.0, D=0.4, H=(0.3, -0.2, 0.4), lam=0.2, T=float(T[r]), dt=0.1, R=R, integrator=integ,
                       seed=21, replica=r)
        ref, smp = orc.run(q, s0[:, r].reshape(3, 1, 1, 1), 21, noise=2)
        assert np.max(np.abs(got[:, r] - ref.reshape(3))) < tol
        assert abs(sums[r] - smp[:, 3].sum()) < 21 * tol


# lattices just within and beyond the sizes that take the per-stage FP32
# kernels: bitwise one trajectory per lattice however its sites are computed --
# a batch replica (always the tile) against the single lattice at the same size,
# and the oracle at a ragged, a flat, a free-boundary and a field lattice
@pytest.mark.parametrize("integ", ["RK4", "RK2_MIDPOINT", "HEUN"])
@pytest.mark.parametrize("L", [8, 47, 48, 49, 64, 65])
def test_fp32_stage_kernels_bitwise(gpu, integ, L):
    if integ == "RK4" and L > 49 or integ == "HEUN" and L not in (8, 64):
        pytest.skip("far from this tableau's size limit")
    kw = dict(J=0.9, D=0.15, H=(0.05, -0.1, 0.2), lam=0.1, dt=0.07, R=3, seed=77, integrator=getattr(gpu, integ))
    s0 = spin_inputs.random_spins(L, L, L, seed=3).astype(np.float32)
    b = gpu.Batch(gpu.Params(1, 1, 1, **kw), [L], [0.7], [s0], chunk_planes=gpu.batch.DEFAULT_TILING)
    lat = gpu.Lattice(gpu.Params(L, L, L, T=0.7, **kw), torch.from_numpy(s0))
    b.step(7)
    lat.step(7)
    torch.cuda.synchronize()
    assert torch.equal(lat.state, b.replica_state(0))


@pytest.mark.parametrize("integ", ["RK4", "RK2_MIDPOINT", "HEUN"])
@pytest.mark.parametrize("shape,precession,hsite,bc", [
    ((129, 151, 1), 1, False, 0), ((1, 1, 700), 0, True, 1), ((45, 37, 27), 1, True, 1), ((57, 56, 55), 0, True, 0)])
def test_fp32_stage_kernels_oracle(gpu, orc, integ, shape, precession, hsite, bc):
    _compare(gpu, orc, shape, 3 * 2e-6, hsite=hsite, precision=32, integrator=getattr(gpu, integ),
             precession=precession, bc=bc)


def test_sample_ring_wraps_and_long_graphs(gpu):
    """Samples read in portions across the ring's end, from intervals replayed
    singly and several to a graph, equal the observables taken step by step."""
    p = gpu.Params(6, 5, 4, J=1.0, D=0.1, H=(0.0, 0.0, 0.2), lam=0.1, T=0.5, dt=0.1, R=2, seed=3)
    s0 = torch.from_numpy(spin_inputs.random_spins(6, 5, 4, seed=3))
    a, b = gpu.Lattice(p, s0), gpu.Lattice(p, s0)
    ring = gpu._binding.SPIN_SAMPLE_RING
    a.step(2 * (ring - 3))
    assert len(a.samples()) == ring - 3
    a.step(2 * 11)
    got = gpu.spin_samples(a.handle, 9)
    for k in range(ring - 3 + 11):
        b.step(2)
    assert torch.equal(a.state, b.state)
    want = b.samples()[-9:]
    assert len(got) == 9 and got == want and got[-1][0] == 2.0 * (ring + 8)


# FP32 gradients whose step terms are added once per step: the order of the
# additions does not depend on the segments, so every K gives the same bits
# (segments of one step, a short last segment, one segment); against the oracle
# with the bounds of test_gpu_adjoint.py; terms of very different size and
# underflowing ones (a loss scaled by 1e-34); a lattice of several blocks with
# idle lanes and rows
@pytest.mark.parametrize("integ,precession", [("RK4", 1), ("RK2_MIDPOINT", 1), ("HEUN", 0)])
def test_adjoint_step_terms(gpu, orc, integ, precession):
    shape, nsteps = (33, 9, 3), 7
    p = gpu.Params(*shape, J=0.9, D=0.25, H=(0.05, -0.1, 0.2), lam=0.1, T=0.8, dt=0.1, R=3, seed=12, precision=32,
                   integrator=getattr(gpu, integ), precession=precession)
    s0 = spin_inputs.random_spins(*shape, seed=11)
    hs = spin_inputs.site_fields(*shape, 0.1, seed=13)

    def grad(K, scale=1.0):
        lat = gpu.Lattice(p, torch.from_numpy(s0), h_site=torch.from_numpy(hs))
        lat.record(K, nsteps)
        lat.step(nsteps)
        g = lat.backward([0.3 * scale, -0.2 * scale, 0.7 * scale], scale, field_grad=True, state_grad=True)
        return np.concatenate([[g["J"], g["D"]], g["H"], g["h"].cpu().numpy().ravel(),
                               g["s0"].double().cpu().numpy().ravel()])

    got = grad(3)
    assert np.array_equal(got, grad(1)) and np.array_equal(got, grad(7))
    ref = orc.adjoint(orc_params(orc, p), as_input(p, s0), nsteps, [0.3, -0.2, 0.7], 1.0, h_site=as_input(p, hs))
    parts = [[ref["J"], ref["D"]], ref["H"], ref["h"], ref["s0"]]
    at = 0
    for r in parts:
        r = np.asarray(r, float).ravel()
        d = got[at:at + r.size] - r
        assert np.max(np.abs(d)) < 1e-5 * np.max(np.abs(r))
        at += r.size
    # scaled by 1e-34 the per-site terms lie below 2^-126 (subnormal, spacing
    # 2^-149): each of the adjoint's roundings is then absolute
    tiny = grad(3, 1e-34)
    n = 5 + 3 * 33 * 9 * 3
    assert np.max(np.abs(tiny[5:n] - 1e-34 * got[5:n])) < 1e-5 * np.max(np.abs(1e-34 * got[5:n])) + 400 * 2.0 ** -149

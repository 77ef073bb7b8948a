"""What a user of the library has it do, as cases to be timed and compared.

A case is one call (or the few calls that belong together) of the public
Python face on a problem that a user's program has prepared: a lattice handle
with its state, a batch of replicas, a recorded run with its gradients, a
Metropolis state, a set of single spins.  ``exact`` states the same problem in
64-bit torch arithmetic (Landau-Lifshitz right-hand side, Runge-Kutta
tableaus, Philox4x64-10 noise, pulse rotation, Metropolis trials) without the
library.

The sizes are those of the repository's own workloads (``spin_inputs.py``,
``bench.py``, ``tests/``); ``draw`` spreads over the ranges around them.
"""
from __future__ import annotations

import math

import torch

import paper_1610_04914_gb300 as sp

DEV = "cuda"
INTEGRATORS = {"rk4": sp.RK4, "rk5": sp.RK5_BUTCHER, "rk2": sp.RK2_MIDPOINT, "heun": sp.HEUN}
STAGES = {"rk4": 4, "rk5": 6, "rk2": 2, "heun": 2}
# flops (FMA = 2) of one site-step: per stage the six-neighbour sum (15), the
# field (7), the two cross products and their sum (24), the stage input and
# the accumulator (12); the renormalisation (9)
RHS_FLOPS = 58
RENORM_FLOPS = 9
# Philox (integer work not counted), Box-Muller and the rotation
PULSE_FLOPS = 80


def _lattice(name, n, **kw):
    c = dict(kind="lattice", name=name, nx=n[0], ny=n[1], nz=n[2], precision=32, integrator="rk4", precession=1,
             bc=0, field=0.0, J=1.0, D=0.05, Hz=0.02, lam=0.01, T=1.0, dt=0.2, R=10, steps=10, ordered=False,
             observe=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest runs: the double-precision reference lattice that
        # trajectories are compared with, one noise interval and M, E read back
        _lattice("small16_fp64", (16, 16, 16), precision=64, D=0.0, Hz=0.1, lam=0.1, dt=0.1, observe=True),
        # a small ragged lattice in a random site field (odd row length, so
        # nothing is aligned), pulses every 5 steps, M and E read back
        _lattice("ragged_field", (45, 37, 27), field=0.01, D=0.02, Hz=0.0, lam=0.05, T=0.8, dt=0.1, R=5, steps=10,
                 observe=True),
        # the throughput workload: one noise interval of the 128^3 lattice
        _lattice("lattice128", (128, 128, 128)),
        # the large lattice: slow equation (precession dropped), odd interval
        _lattice("overdamped256", (256, 256, 256), precession=0, D=0.0, Hz=0.01, lam=1.0, T=1.2, R=5, steps=5),
        # the paper's 64^3 particle: free boundaries, RK2 midpoint, a pulse
        # every other step, ordered start; the samples of the run read back
        _lattice("particle64_rk2", (64, 64, 64), integrator="rk2", precession=0, bc=1, D=0.0, Hz=0.0, dt=4.0, R=2,
                 steps=20, ordered=True, observe=True),
        # the paper's higher-order integrator (Butcher RK5) on the 128^3 lattice
        _lattice("lattice128_rk5", (128, 128, 128), integrator="rk5", dt=0.1),
        # the same lattice in double precision, for a run to be trusted to 1e-13
        _lattice("lattice128_fp64", (128, 128, 128), precision=64, dt=0.1, R=4, steps=4),
        # an ensemble over sizes and temperatures in one batch
        dict(kind="batch", name="batch96", nrep=96, Lmin=16, Lmax=64, J=1.0, D=0.02, lam=0.02, dt=0.2, R=10,
             steps=10, integrator="rk4"),
        # gradients with respect to J, D, H, every site field and the initial
        # state through 20 recorded steps, a checkpoint every 10
        dict(kind="adjoint", name="adjoint64", nx=64, ny=64, nz=64, integrator="rk4", D=0.05, field=0.01, lam=0.05,
             T=0.8, dt=0.1, R=10, K=10, steps=20),
        # the comparison method: checkerboard Metropolis sweeps
        dict(kind="metropolis", name="metropolis128", nx=128, ny=128, nz=128, precision=32, bc=0, T=1.0, sweeps=4),
        # single spins in a field, pulse noise, equilibrium averages (Langevin
        # function): every replica of a grid of temperatures in one launch
        dict(kind="single", name="single_langevin", nrep=131072, integrator="rk5", noise=1, D=0.0, Hx=0.0, Hz=1.0,
             lam=0.01, T=1.0, dt=0.25, R=40, steps=400, precision=32),
        # the conventional scheme it is compared with: Heun, a new rectangular
        # noise field every step
        dict(kind="single", name="single_heun_rect", nrep=32768, integrator="heun", noise=2, D=0.0, Hx=0.0, Hz=1.0,
             lam=0.01, T=1.0, dt=0.04, R=1, steps=200, precision=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides(rng, lo, hi, most, even=False):
    """Three sides, log-uniform, odd ones among them, at most `most` sites."""
    while True:
        n = [_log_int(rng, lo, hi) for _ in range(3)]
        if rng.random() < 0.4:
            n = [n[0]] * 3   # cubes are what most runs use
        if even:
            n = [v + (v & 1) for v in n]
        if n[0] * n[1] * n[2] <= most:
            return n


def draw(rng):
    kind = rng.choice(["lattice", "lattice", "lattice", "lattice64", "batch", "adjoint", "metropolis", "single"])
    if kind in ("lattice", "lattice64"):
        fp64 = kind == "lattice64"
        n = _sides(rng, 8, 128 if fp64 else 256, 1 << 20 if fp64 else 1 << 24)
        integ = rng.choice(["rk4", "rk4", "rk4", "rk2", "heun", "rk5"])
        prec = 1 if rng.random() < 0.7 else 0
        R = rng.choice([2, 4, 5, 10]) if not fp64 else rng.choice([2, 4, 5])
        return _lattice("", n, precision=64 if fp64 else 32, integrator=integ, precession=prec,
                        bc=1 if rng.random() < 0.3 else 0, field=0.01 if rng.random() < 0.25 else 0.0,
                        D=rng.choice([0.0, 0.02, 0.05]), Hz=rng.choice([0.0, 0.02, 0.1]),
                        lam=rng.choice([0.01, 0.05, 0.1]), T=round(rng.uniform(0.2, 1.6), 3),
                        dt=0.1, R=R, steps=R * rng.choice([1, 2]) if not fp64 else R, observe=rng.random() < 0.3)
    if kind == "batch":
        lo = rng.choice([8, 12, 16, 24])
        return dict(kind="batch", nrep=_log_int(rng, 8, 96), Lmin=lo, Lmax=rng.choice([32, 48, 64]), J=1.0, D=0.02,
                    lam=0.02, dt=0.1, R=10, steps=10, integrator=rng.choice(["rk4", "rk4", "rk2", "heun"]))
    if kind == "adjoint":
        n = _sides(rng, 12, 72, 300000)
        return dict(kind="adjoint", nx=n[0], ny=n[1], nz=n[2], integrator=rng.choice(["rk4", "rk4", "rk2", "heun"]),
                    D=0.05, field=0.01, lam=0.05, T=0.8, dt=0.1, R=rng.choice([5, 10]), K=rng.choice([5, 10]),
                    steps=rng.choice([10, 20]))
    if kind == "metropolis":
        bc = 1 if rng.random() < 0.3 else 0
        n = _sides(rng, 16, 192, 1 << 22, even=bc == 0)
        return dict(kind="metropolis", nx=n[0], ny=n[1], nz=n[2], precision=32, bc=bc,
                    T=round(rng.uniform(0.3, 1.6), 3), sweeps=rng.choice([1, 2, 4]))
    noise = rng.choice([1, 1, 2])
    R = rng.choice([6, 20, 40]) if noise == 1 else rng.choice([1, 4])
    return dict(kind="single", nrep=_log_int(rng, 1000, 200000), integrator=rng.choice(["rk5", "rk5", "rk4", "heun"]),
                noise=noise, D=0.0, Hx=0.0, Hz=1.0, lam=0.01, T=round(rng.uniform(0.1, 1.0), 3),
                dt=rng.choice([0.04, 0.1, 0.2]), R=R, steps=R * max(1, 240 // R), precision=32)


# ---- inputs ---------------------------------------------------------------

def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + stream * 7919 + 12345) % (1 << 62))
    return g


def _unit(shape, seed, stream, ordered=False):
    """Unit spins (3, ...) uniform on the sphere; ordered: along z with the
    spread of a cold start."""
    v = torch.randn((3,) + tuple(shape), generator=_gen(seed, stream), device=DEV, dtype=torch.float32)
    if ordered:
        v = 0.05 * v
        v[2] += 1.0
    v = v.double()
    return v / v.square().sum(0, keepdim=True).sqrt()


def _noise_seed(seed):
    return (int(seed) * 2654435761 + 17) % (1 << 63)


def _lattice_params(c, seed):
    return sp.Params(c["nx"], c["ny"], c["nz"], J=c["J"], D=c["D"], H=(0.0, 0.0, c["Hz"]), lam=c["lam"], T=c["T"],
                     dt=c["dt"], R=c["R"], integrator=INTEGRATORS[c["integrator"]], precession=c["precession"],
                     seed=_noise_seed(seed), precision=c["precision"], bc=c["bc"])


def _lattice_inputs(c, seed):
    dt = torch.float64 if c["precision"] == 64 else torch.float32
    shape = (c["nz"], c["ny"], c["nx"])
    s0 = _unit(shape, seed, 1, c["ordered"]).to(dt)
    h = None
    if c["field"]:
        h = (c["field"] * torch.randn((3,) + shape, generator=_gen(seed, 2), device=DEV, dtype=torch.float32)).to(dt)
    return s0, h


def _adjoint_params(c, seed):
    return sp.Params(c["nx"], c["ny"], c["nz"], J=1.0, D=c["D"], H=(0.0, 0.0, 0.0), lam=c["lam"], T=c["T"],
                     dt=c["dt"], R=c["R"], integrator=INTEGRATORS[c["integrator"]], seed=_noise_seed(seed),
                     precision=32)


def _adjoint_inputs(c, seed):
    shape = (c["nz"], c["ny"], c["nx"])
    h = c["field"] * torch.randn((3,) + shape, generator=_gen(seed, 2), device=DEV, dtype=torch.float32)
    return _unit(shape, seed, 1, True).float(), h


def _batch_plan(c, seed):
    """Replica sides over {16, 24, 32, 48, 64} within the case's range (with
    an odd side where the range starts below 16) and temperatures."""
    sides = [v for v in (8, 11, 12, 16, 24, 32, 48, 64) if c["Lmin"] <= v <= c["Lmax"]]
    n = c["nrep"]
    L = [sides[(5 * r + r // len(sides)) % len(sides)] for r in range(n)]
    T = [0.2 + 1.8 * ((r * 0.6180339887 + (seed % 97) / 97.0) % 1.0) for r in range(n)]
    return L, T


def _batch_inputs(c, seed):
    L, T = _batch_plan(c, seed)
    total = sum(l ** 3 for l in L)
    return L, T, _unit((total,), seed, 1).float()


def _single_inputs(c, seed):
    T = [c["T"] * (0.5 + r / c["nrep"]) for r in range(c["nrep"])]
    return T, _unit((c["nrep"],), seed, 1).float()


def _single_params(c, seed):
    return sp.Params(1, 1, 1, J=0.0, D=c["D"], H=(c["Hx"], 0.0, c["Hz"]), lam=c["lam"], T=c["T"], dt=c["dt"],
                     R=c["R"], integrator=INTEGRATORS[c["integrator"]], noise=c["noise"], seed=_noise_seed(seed),
                     precision=c["precision"])


def _mc_params(c):
    return sp.Params(c["nx"], c["ny"], c["nz"], J=1.0, T=c["T"], bc=c["bc"], precision=c["precision"])


def prepare(case, seed):
    c = case
    if c["kind"] == "lattice":
        s0, h = _lattice_inputs(c, seed)
        return {"case": c, "lat": sp.Lattice(_lattice_params(c, seed), s0, h_site=h)}
    if c["kind"] == "batch":
        L, T, flat = _batch_inputs(c, seed)
        p = sp.Params(1, 1, 1, J=c["J"], D=c["D"], H=(0.0, 0.0, 0.0), lam=c["lam"], dt=c["dt"], R=c["R"],
                      integrator=INTEGRATORS[c["integrator"]], seed=_noise_seed(seed), precision=32)
        return {"case": c, "batch": sp.Batch(p, L, T, flat.cpu().numpy(), use_cache=False)}
    if c["kind"] == "adjoint":
        s0, h = _adjoint_inputs(c, seed)
        p = _adjoint_params(c, seed)
        lat = sp.Lattice(p, s0, h_site=h)
        # the recording store, the backward workspace and the gradients are
        # kept by a program that takes many gradients
        n = (3, p.nz, p.ny, p.nx)
        return {"case": c, "lat": lat, "s0": s0,
                "store": torch.empty(sp.spin_record_store_size(p, c["K"], c["steps"]) // 8 + 1, dtype=torch.float64,
                                     device=DEV),
                "ws": torch.empty(sp.spin_backward_workspace_size(p, c["K"]) // 8 + 32, dtype=torch.float64,
                                  device=DEV),
                "gh": torch.empty(n, dtype=torch.float64, device=DEV),
                "gs": torch.empty(n, dtype=torch.float32, device=DEV)}
    if c["kind"] == "metropolis":
        shape = (c["nz"], c["ny"], c["nx"])
        return {"case": c, "p": _mc_params(c), "state": _unit(shape, seed, 1, True).float().contiguous(),
                "seed": _noise_seed(seed), "sweep": 0, "acc": torch.zeros(1, dtype=torch.int64, device=DEV)}
    T, s = _single_inputs(c, seed)
    return {"case": c, "spins": sp.SingleSpins(_single_params(c, seed), T, s)}


def run(state):
    c = state["case"]
    if c["kind"] == "lattice":
        lat = state["lat"]
        lat.step(c["steps"])
        if not c["observe"]:
            return {"state": lat.state}
        M, E = lat.observables()
        # the samples taken at the ends of this call's intervals
        rec = [list(r[1:]) for r in lat.samples()[-(c["steps"] // c["R"]):]]
        return {"state": lat.state, "M_E": torch.tensor(M + [E], dtype=torch.float32),
                "samples": torch.tensor(rec, dtype=torch.float32)}
    if c["kind"] == "batch":
        b = state["batch"]
        b.step(c["steps"])
        return {"state": b.state}
    if c["kind"] == "adjoint":
        # one gradient evaluation: restart from s0, record, run, loss
        # E + |M - (0, 0, 1/2)|^2 at the final state, gradients
        lat = state["lat"]
        lat.state.copy_(state["s0"])
        lat.set_step(0)
        sp.spin_record_begin(lat.handle, c["K"], c["steps"], state["store"])
        lat.step(c["steps"])
        M, E = lat.observables()
        dM = [2.0 * M[0], 2.0 * M[1], 2.0 * (M[2] - 0.5)]
        gJ, gD, gH = sp.spin_backward(lat.handle, dM, 1.0, state["ws"], state["gh"], state["gs"])
        sp.spin_record_end(lat.handle)
        # the site field is held in float32, so is its gradient
        return {"state": lat.state, "J": gJ, "D": gD, "H": torch.tensor(gH, dtype=torch.float32), "h": state["gh"].float(), "s0": state["gs"]}
    if c["kind"] == "metropolis":
        sp.spin_metropolis_sweeps(state["p"], state["state"], c["sweeps"], mc_seed=state["seed"],
                                  sweep0=state["sweep"], accepted=state["acc"])
        state["sweep"] += c["sweeps"]
        return {"state": state["state"], "accepted": state["acc"]}
    s = state["spins"]
    s.run(c["steps"], average=True)
    return {"state": s.state, "sz_sum": s.sz_sum.float(), "sz_count": s.sz_count}


def work(case):
    c = case
    if c["kind"] == "lattice":
        n = c["nx"] * c["ny"] * c["nz"]
        w = c["precision"] // 8
        per = STAGES[c["integrator"]] * RHS_FLOPS + RENORM_FLOPS
        return {"bytes": n * w * (6 + (3 if c["field"] else 0)),
                "flops": n * (c["steps"] * per + c["steps"] // c["R"] * PULSE_FLOPS)}
    if c["kind"] == "batch":
        n = sum(l ** 3 for l in _batch_plan(c, 0)[0])
        per = STAGES[c["integrator"]] * RHS_FLOPS + RENORM_FLOPS
        return {"bytes": 24 * n, "flops": n * (c["steps"] * per + c["steps"] // c["R"] * PULSE_FLOPS)}
    if c["kind"] == "adjoint":
        n = c["nx"] * c["ny"] * c["nz"]
        per = STAGES[c["integrator"]] * RHS_FLOPS + RENORM_FLOPS
        # in: s0 and the field; out: the state, dL/dh (FP64) and dL/ds0; the
        # transposed step costs about twice the forward step, run once more
        return {"bytes": n * (12 + 12 + 12 + 24 + 12), "flops": n * c["steps"] * per * 4}
    if c["kind"] == "metropolis":
        n = c["nx"] * c["ny"] * c["nz"]
        return {"bytes": 24 * n, "flops": 90 * n * c["sweeps"]}
    n = c["nrep"]
    per = STAGES[c["integrator"]] * 42 + RENORM_FLOPS
    draws = c["steps"] // c["R"]
    return {"bytes": n * (24 + 8 + 16 + 16), "flops": n * (c["steps"] * per + draws * PULSE_FLOPS)}


# ---- the same in 64-bit torch ---------------------------------------------

_RK = {
    "rk4": ([[], [0.5], [0.0, 0.5], [0.0, 0.0, 1.0]], [1 / 6, 1 / 3, 1 / 3, 1 / 6]),
    "rk2": ([[], [0.5]], [0.0, 1.0]),
    "heun": ([[], [1.0]], [0.5, 0.5]),
    "rk5": ([[], [1 / 4], [1 / 8, 1 / 8], [0.0, -1 / 2, 1.0], [3 / 16, 0.0, 0.0, 9 / 16],
             [-3 / 7, 2 / 7, 12 / 7, -12 / 7, 8 / 7]], [7 / 90, 0.0, 32 / 90, 12 / 90, 32 / 90, 7 / 90]),
}
_M32 = 0xFFFFFFFF


def _i64(v):
    v &= (1 << 64) - 1
    return v - (1 << 64) if v >> 63 else v


def _hi(x):
    return (x >> 32) & _M32


def _mulhi(a, m):
    m0, m1 = m & _M32, m >> 32
    a0, a1 = a & _M32, _hi(a)
    t = a1 * m0 + _hi(a0 * m0)
    u = a0 * m1 + (t & _M32)
    return a1 * m1 + _hi(t) + _hi(u)


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x64-10 on int64 tensors (bit patterns of the unsigned words)."""
    A, B = 0xD2E7470EE14C6C93, 0xCA5A826395121157
    for r in range(10):
        ka, kb = _i64(k0 + r * 0x9E3779B97F4A7C15), _i64(k1 + r * 0xBB67AE8584CAA73B)
        ha, la, hb, lb = _mulhi(c0, A), c0 * _i64(A), _mulhi(c2, B), c2 * _i64(B)
        c0, c1, c2, c3 = hb ^ c1 ^ ka, lb, ha ^ c3 ^ kb, la
    return c0, c1, c2, c3


def _u01(w):
    return (((w >> 11) & ((1 << 53) - 1)).double() + 0.5) * 2.0 ** -53


def _gauss(site, k, replica, seed):
    z = torch.zeros_like(site)
    w = _philox(site, z + k, z + replica, z, seed, 0x6E6F697365)
    u = [_u01(v) for v in w]
    r0, r2 = (-2 * u[0].log()).sqrt(), (-2 * u[2].log()).sqrt()
    return torch.stack([r0 * (2 * math.pi * u[1]).cos(), r0 * (2 * math.pi * u[1]).sin(),
                        r2 * (2 * math.pi * u[3]).cos()])


def _cross(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])


def _rotate(s, phi):
    a = phi.square().sum(0).sqrt()
    n = phi / a.clamp(min=1e-300)
    ns = (n * s).sum(0)
    return s * a.cos() + _cross(n, s) * a.sin() + n * (ns * (1 - a.cos()))


def _neighbours(s, bc):
    out = torch.zeros_like(s)
    for d in (1, 2, 3):
        for shift in (1, -1):
            t = torch.roll(s, shift, d)
            if bc:
                t = t.clone()
                t.select(d, 0 if shift == 1 else s.shape[d] - 1).zero_()
            out = out + t
    return out


def _field(s, nn, J, D, H):
    return J * nn + H + torch.stack([torch.zeros_like(s[2]), torch.zeros_like(s[2]), 2 * D * s[2]])


def _rk_step(s, rhs, dt, integ):
    a, b = _RK[integ]
    K = []
    for j in range(len(b)):
        x = s
        for l, v in enumerate(a[j]):
            if v:
                x = x + v * K[l]
        K.append(dt * rhs(x))
    y = s
    for w, k in zip(b, K):
        if w:
            y = y + w * k
    return y / y.square().sum(0, keepdim=True).sqrt()


def _llg(x, Heff, lam, precession, extra=None):
    a = _cross(x, Heff)
    b = _cross(x, a)
    if not precession:
        return -lam * b
    return (a if extra is None else a + _cross(x, extra)) - lam * b


def _lattice_run(s, J, D, H, c, seed, steps, R, noise_T, replica=0, samples=None, bc=0, precession=1, site0=None):
    n = s[0].numel()
    sites = torch.arange(n, device=s.device, dtype=torch.int64)
    sigma = math.sqrt(2 * c["lam"] * noise_T * R * abs(c["dt"]))
    for m in range(1, steps + 1):
        s = _rk_step(s, lambda x: _llg(x, _field(x, _neighbours(x, bc), J, D, H), c["lam"], precession), c["dt"],
                     c["integrator"])
        if m % R == R // 2:
            g = _gauss(sites, (m - 1) // R, replica, seed).reshape(s.shape)
            s = _rotate(s, sigma * g)
        if samples is not None and m % R == 0:
            samples.append(s)
    return s


def _observables(s, J, D, H, bc):
    N = s[0].numel()
    M = s.reshape(3, -1).mean(1)
    e = -0.5 * J * (s * _neighbours(s, bc)).sum() - D * s[2].square().sum() - (H * s).sum()
    return M, e / N


def exact(case, seed):
    c = case
    if c["kind"] == "lattice":
        s, h = _lattice_inputs(c, seed)
        s = s.double()
        H = torch.tensor([0.0, 0.0, c["Hz"]], device=DEV, dtype=torch.float64).reshape(3, 1, 1, 1)
        if h is not None:
            H = H + h.double()
        states = []
        s = _lattice_run(s, c["J"], c["D"], H, c, _noise_seed(seed), c["steps"], c["R"], c["T"], samples=states,
                         bc=c["bc"], precession=c["precession"])
        if not c["observe"]:
            return {"state": s}
        M, E = _observables(s, c["J"], c["D"], H, c["bc"])
        rec = []
        for q in states:
            m, e = _observables(q, c["J"], c["D"], H, c["bc"])
            rec.append(m.tolist() + [float(e)])
        return {"state": s, "M_E": torch.tensor(M.tolist() + [float(E)], dtype=torch.float64),
                "samples": torch.tensor(rec, dtype=torch.float64)}
    if c["kind"] == "batch":
        L, T, flat = _batch_inputs(c, seed)
        flat, at = flat.double(), 0
        H = torch.zeros((3, 1, 1, 1), device=DEV, dtype=torch.float64)
        out = torch.empty_like(flat)
        if c["nrep"] > 128:
            return None
        for r, (l, t) in enumerate(zip(L, T)):
            s = flat[:, at:at + l ** 3].reshape(3, l, l, l)
            s = _lattice_run(s, c["J"], c["D"], H, c, _noise_seed(seed), c["steps"], c["R"], t, replica=r)
            out[:, at:at + l ** 3] = s.reshape(3, -1)
            at += l ** 3
        return {"state": out}
    if c["kind"] == "adjoint":
        s0, h = _adjoint_inputs(c, seed)
        leaf = lambda v: torch.as_tensor(v, dtype=torch.float64, device=DEV).clone().requires_grad_(True)  # noqa: E731
        J, D, Hu, hs, x0 = leaf(1.0), leaf(c["D"]), leaf([0.0, 0.0, 0.0]), leaf(h), leaf(s0)
        H = Hu.reshape(3, 1, 1, 1) + hs
        s = _lattice_run(x0, J, D, H, c, _noise_seed(seed), c["steps"], c["R"], c["T"])
        M, E = _observables(s, J, D, H, 0)
        target = torch.tensor([0.0, 0.0, 0.5], device=DEV, dtype=torch.float64)
        g = torch.autograd.grad(E + (M - target).square().sum(), [J, D, Hu, hs, x0])
        return {"state": s.detach(), "J": float(g[0]), "D": float(g[1]), "H": g[2], "h": g[3], "s0": g[4]}
    if c["kind"] == "metropolis":
        return {"state": _metropolis(c, seed), "accepted": None}
    T, s = _single_inputs(c, seed)
    return _single(c, seed, torch.tensor(T, dtype=torch.float64, device=DEV), s.double())


def _metropolis(c, seed):
    shape = (c["nz"], c["ny"], c["nx"])
    s = _unit(shape, seed, 1, True).float().double()
    site = torch.arange(s[0].numel(), device=DEV, dtype=torch.int64)
    zyx = [torch.arange(n, device=DEV) for n in shape]
    colour = ((zyx[0][:, None, None] + zyx[1][None, :, None] + zyx[2][None, None, :]) & 1)
    length, zero = 1.55 * math.sqrt(c["T"] / 6.0), torch.zeros_like(site)
    for sweep in range(c["sweeps"]):
        u = [_u01(w).reshape(shape) for w in _philox(site, zero + sweep, zero, zero, _noise_seed(seed), 0x6D6F6E7465)]
        cz = 2 * u[0] - 1
        st = (1 - cz * cz).sqrt()
        v = torch.stack([st * (2 * math.pi * u[1]).cos(), st * (2 * math.pi * u[1]).sin(), cz])
        for col in (0, 1):
            new = s + length * v
            new = new / new.square().sum(0, keepdim=True).sqrt()
            nn = _neighbours(s, c["bc"])
            dE = -((new - s) * nn).sum(0)
            ok = (colour == col) & ((dE <= 0) | (u[2] < (-dE / c["T"]).exp()))
            s = torch.where(ok, new, s)
    return s


def _single(c, seed, T, s):
    rep = torch.arange(c["nrep"], device=DEV, dtype=torch.int64)
    zero = torch.zeros_like(rep)
    H = torch.tensor([c["Hx"], 0.0, c["Hz"]], device=DEV, dtype=torch.float64).reshape(3, 1).expand_as(s)
    Dt = c["R"] * abs(c["dt"])
    rect = c["noise"] == 2
    scale = (2 * c["lam"] * T / Dt).sqrt() if rect else (2 * c["lam"] * T * Dt).sqrt()
    acc, z = torch.zeros_like(s[2]), None

    def gauss(k):
        w = _philox(zero, zero + k, rep, zero, _noise_seed(seed), 0x6E6F697365)
        u = [_u01(v) for v in w]
        r0, r2 = (-2 * u[0].log()).sqrt(), (-2 * u[2].log()).sqrt()
        return torch.stack([r0 * (2 * math.pi * u[1]).cos(), r0 * (2 * math.pi * u[1]).sin(),
                            r2 * (2 * math.pi * u[3]).cos()])

    for m in range(1, c["steps"] + 1):
        if rect and (m - 1) % c["R"] == 0:
            z = scale * gauss((m - 1) // c["R"])
        s = _rk_step(s, lambda x: _llg(x, _field(x, torch.zeros_like(x), 0.0, c["D"], H), c["lam"], 1, z), c["dt"],
                     c["integrator"])
        if not rect and m % c["R"] == c["R"] // 2:
            s = _rotate(s, scale * gauss((m - 1) // c["R"]))
        if m % c["R"] == 0:
            acc = acc + s[2]
    return {"state": s, "sz_sum": acc, "sz_count": None}

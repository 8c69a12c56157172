"""Performance cases of the particle-in-cell framework.

Each case is one pass of a program that uses the framework: a run of some steps
whose particles and fields are then read, a sweep with its gradient, an
ensemble, a loop that couples through host memory.  Sizes follow the mini-apps
of the benchmark and the tests (Landau damping, two-stream and bump-on-tail,
Penning trap, uniform plasma, ensembles) and generic odd ones.

Inputs are drawn on the GPU from the seed.  `exact` restates the scheme in
64-bit torch, with the library's documented conventions (cell-centred grid,
cloud-in-cell shape, spectral field, drift-kick-drift), and takes gradients
with torch's autograd.
"""
import math
import random
import types

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2205_11052_gb300 import capi
from paper_2205_11052_gb300.autograd import final_field_energy
from paper_2205_11052_gb300.batch import Ensemble
from paper_2205_11052_gb300.shard import sharded_simulation
from paper_2205_11052_gb300.sim import Simulation

FIXED, MOVE, PARAMS = 1, 2, 4      # option bits: fixed-point deposit, random move, parameter gradients

# physics of each mini-app: box length, perturbation, fields
FAMILY = {
    "landau": dict(L=4 * math.pi, k=0.5, alpha=0.05, B=(0.0, 0.0, 0.0), wz2=0.0),
    "two_stream": dict(L=4 * math.pi, k=0.5, alpha=0.01, B=(0.0, 0.0, 0.0), wz2=0.0),
    "bump": dict(L=20 * math.pi, k=0.1, alpha=0.05, B=(0.0, 0.0, 0.0), wz2=0.0),
    "penning": dict(L=20.0, B=(0.0, 0.0, 5.0), wz2=1.0),
    "uniform": dict(L=4 * math.pi, B=(0.0, 0.0, 0.0), wz2=0.0),
}


def _case(name, kind, family, grid, particles, steps, options=FIXED, sort_period=4, diag_every=1, guard=0, tile=0,
          stray=0.0, keep=0, mix=0, dt=0.05):
    c = dict(kind=kind, family=family, nx=grid[0], ny=grid[1], nz=grid[2], particles=particles, steps=steps,
             options=options, sort_period=sort_period, diag_every=diag_every, guard=guard, tile=tile, stray=stray,
             keep=keep, mix=mix, dt=dt)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a small run with every setting at its default, as in the tests and a first try: launches and latency
        _case("landau16_defaults", "run", "landau", (16, 16, 16), 16 ** 3 * 8, 20, options=0, sort_period=0),
        # odd sizes on every axis, an odd particle count, FP32 deposit, no diagnostics
        _case("two_stream_ragged", "run", "two_stream", (45, 28, 36), 300_007, 10, options=0, sort_period=2,
              diag_every=0),
        # the bump-on-tail workload of the benchmark: an ordinary run
        _case("bump64", "run", "bump", (64, 64, 64), 64 ** 3 * 16, 20),
        # the benchmark's headline workload
        _case("landau128", "run", "landau", (128, 128, 128), 128 ** 3 * 64, 20),
        # the trap: strongly non-uniform occupancy, Boris rotation and quadrupole, three guard layers
        _case("penning256", "run", "penning", (256, 256, 256), 130_000_000, 10, sort_period=2, guard=3),
        # the strong-scaling cases' few particles per cell and dt = h/2 on a large grid
        _case("landau256_8ppc", "run", "landau", (256, 256, 256), 256 ** 3 * 8, 8, dt=2 * math.pi / 256),
        # the uniform plasma test (random moves instead of the push)
        _case("uniform128_move", "run", "uniform", (128, 128, 128), 128 ** 3 * 16, 8, options=FIXED | MOVE),
        # the cycle by separate calls, as a particle-sharded run drives it on each rank
        _case("split64", "split", "landau", (64, 64, 64), 64 ** 3 * 64, 8, diag_every=0),
        # gradient of the final field energy through the autograd function, checkpointed, at the benchmark's size
        _case("adjoint_bump64", "adjoint", "bump", (64, 64, 64), 64 ** 3 * 16, 20, keep=5),
        # a small gradient in the trap, with the field parameters' gradients
        _case("adjoint_trap24", "adjoint", "penning", (24, 24, 24), 60_001, 12, options=FIXED | PARAMS, keep=4,
              sort_period=2),
        # an ensemble of uneven Landau runs (16, 24, 32 or 48 cells an axis, 8 to 64 particles per cell)
        _case("ensemble24", "ensemble", "landau", (0, 0, 0), 0, 8, mix=24_001),
        # a program that couples through page-locked host memory: load, a few steps, records and particles back
        _case("host_loop96", "host", "landau", (96, 96, 96), 8_000_000, 4),
    ]


def _axis(rng, most):
    return max(2, int(round(math.exp(rng.uniform(math.log(8), math.log(most + 0.49))))))


def draw(rng):
    """One more case: any kind, grids of 8 to 256 nodes an axis (cubes and ragged boxes), about a thousand to
    fifty million particles, the settings the autotuner and the benchmark choose between."""
    kind = rng.choice(["run", "run", "run", "run", "split", "adjoint", "ensemble", "host"])
    steps = rng.randrange(2, 21)
    sort_period = rng.choice([0, 2, 4, 8])
    if kind == "ensemble":
        return _case("", kind, "landau", (0, 0, 0), 0, min(steps, 8), options=rng.choice([FIXED, FIXED, 0]),
                     sort_period=sort_period, tile=rng.choice([0, 4]), diag_every=rng.choice([0, 1]),
                     mix=rng.randrange(2, 25) * 1000 + rng.randrange(1000))
    most = {"run": 256, "split": 128, "adjoint": 64, "host": 128}[kind]
    if rng.random() < 0.4:
        n = _axis(rng, most)
        grid = (n, n, n)
    else:
        grid = tuple(_axis(rng, most) for _ in range(3))
    top = {"run": 50e6, "split": 20e6, "adjoint": 4e6, "host": 8e6}[kind]
    # 2 to 100 particles per cell and an odd remainder
    ppc = math.exp(rng.uniform(math.log(2), math.log(100)))
    particles = min(int(grid[0] * grid[1] * grid[2] * ppc) + rng.randrange(100), int(top) + rng.randrange(100))
    if kind == "adjoint":
        family = rng.choice(["bump", "landau", "penning"])
        dt = _dt(family, grid)
        options = FIXED | (PARAMS if family == "penning" and rng.random() < 0.5 else 0)
        return _case("", kind, family, grid, particles, steps, options=options, sort_period=sort_period,
                     keep=rng.randrange(2, 11), dt=dt)
    family = rng.choice(["landau", "landau", "two_stream", "bump", "penning", "uniform"])
    options = rng.choice([FIXED, FIXED, 0])
    if family == "uniform" and kind != "split" and rng.random() < 0.5:
        options |= MOVE
    # the penning bunch takes three guard layers in the benchmark; the autotuner tries one and two, tiles of 8 and 4
    guard = 3 if family == "penning" else rng.choice([0, 0, 1])
    stray = 1e-3 if kind == "run" and rng.random() < 0.25 else 0.0
    return _case("", kind, family, grid, particles, steps, options=options, sort_period=sort_period,
                 diag_every=rng.choice([0, 1]), guard=guard, tile=rng.choice([0, 0, 0, 4]), stray=stray,
                 dt=_dt(family, grid))


# ------------------------------------------------------------------ inputs

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed))
    return g


def _cosine(u, L, alpha, k):
    """Samples of 1 + alpha cos(k x) on [0, L) by Newton iteration on the inverse of its distribution."""
    x = u * L
    for _ in range(6):
        x = (x - (x + (alpha / k) * torch.sin(k * x) - u * L) / (1 + alpha * torch.cos(k * x))).clamp_(0, L)
    return torch.where(x >= L, torch.zeros_like(x), x)


def _phase_space(family, n, gen, alpha=None):
    """(x, v): (n, 3) float64 particles of a mini-app."""
    f = FAMILY[family]
    kw = dict(generator=gen, dtype=torch.float64, device=gen.device)
    x = torch.empty((n, 3), dtype=torch.float64, device=gen.device)
    v = torch.randn((n, 3), **kw)
    for d in range(3):
        if family == "penning":
            x[:, d] = torch.remainder(0.5 * f["L"] + (1.0, 1.0, 2.0)[d] * torch.randn(n, **kw), f["L"])
        else:
            u = torch.rand(n, **kw)
            if family == "landau" or (family in ("two_stream", "bump") and d == 2):
                x[:, d] = _cosine(u, f["L"], alpha if alpha is not None else f["alpha"], f["k"])
            else:
                x[:, d] = u * f["L"]
    if family == "two_stream":
        v *= 0.1
        v[:, 2] += torch.where(torch.rand(n, **kw) < 0.5, math.pi / 2, -math.pi / 2)
    if family == "bump":
        beam = torch.rand(n, **kw) < 0.1
        v[:, 2] = torch.where(beam, 4.0 + 0.3 * v[:, 2], v[:, 2])
    return x, v


def _charge(family):
    return -1562.5 if family == "penning" else -FAMILY[family]["L"] ** 3


def _dt(family, grid):
    """0.05, and at most a cell per unit speed on fine grids."""
    return min(0.05, FAMILY[family]["L"] / max(grid))


def _members(case):
    """[(n, particles, alpha)] of an ensemble: part of the case, not of the seed."""
    r = random.Random(case["mix"])
    out = []
    for _ in range(case["mix"] // 1000):
        n = r.choice([16, 24, 32, 48])
        out.append((n, n ** 3 * r.randint(8, 64) + r.randint(0, 999), r.uniform(0.01, 0.1)))
    return out


def _mode(case):
    return dict(mode=(0, 0, 1), mode_comp=2) if case["family"] != "landau" else dict(mode=(1, 0, 0), mode_comp=0)


def _settings(case):
    return dict(sort_period=case["sort_period"], options=case["options"], diag_every=case["diag_every"],
                guard=case["guard"], tile=(case["tile"],) * 3, **_mode(case))


def prepare(case, seed):
    f = FAMILY[case["family"]]
    gen = _gen(seed)
    if case["kind"] == "ensemble":
        members, parts = [], []
        for n, count, alpha in _members(case):
            x, v = _phase_space("landau", count, gen, alpha)
            parts.append((x, v))
            members.append((n, f["L"], x.cpu().numpy(), v.cpu().numpy(), -f["L"] ** 3))
        ens = Ensemble(members, dt=0.05, **_settings(dict(case, guard=0)))
        return dict(case=case, ens=ens)
    grid = (case["nx"], case["ny"], case["nz"])
    x, v = _phase_space(case["family"], case["particles"], gen)
    base = dict(n=grid, L=(f["L"],) * 3, n_particles=case["particles"], dt=case["dt"], Q=_charge(case["family"]),
                B=f["B"], wz2=f["wz2"])
    if case["kind"] == "split":
        w = types.SimpleNamespace(x=x, v=v, q_over_m=-1.0, **_mode(case), **base)
        extra = {k: s for k, s in _settings(case).items() if k not in ("sort_period", "mode", "mode_comp")}
        sim, stepper, _ = sharded_simulation(w, 0, 1, sort_period=max(1, case["sort_period"]), **extra)
        return dict(case=case, sim=sim, stepper=stepper)
    sim = Simulation(seed=int(seed), stray_rebin=case["stray"], **base, **_settings(case))
    if case["kind"] == "adjoint":
        return dict(case=case, sim=sim, x=x.requires_grad_(), v=v.requires_grad_())
    if case["kind"] == "host":
        pinned = [t.cpu().pin_memory() for t in (x, v, x, v)]
        return dict(case=case, sim=sim, pinned=pinned)
    sim.load(x, v)
    return dict(case=case, sim=sim)


# ------------------------------------------------------------------ one pass

def _fields(sim):
    """The charge density and the field, copied to device tensors of the caller."""
    nx, ny, nz = sim.n
    rho = torch.empty((nz, ny, nx), dtype=torch.float32, device=sim.device)
    E = torch.empty((nz, ny, nx, 4), dtype=torch.float32, device=sim.device)
    capi.pic_get_field(sim.handle, rho.data_ptr(), E.data_ptr(), True)
    return rho, E


def run(state):
    case = state["case"]
    if case["kind"] == "ensemble":
        ens = state["ens"]
        ens.step(case["steps"])
        n = sum(ens.counts)
        x = torch.empty((n, 3), dtype=torch.float64, device=ens.device)
        v = torch.empty((n, 3), dtype=torch.float64, device=ens.device)
        capi.pic_batch_get_particles(ens.handle, x.data_ptr(), v.data_ptr(), True)
        return dict(x=x, v=v)
    sim = state["sim"]
    if case["kind"] == "adjoint":
        J = final_field_energy(state["x"], state["v"], sim, case["steps"], (1.0, 1.0, 1.0), case["keep"])
        gx, gv = torch.autograd.grad(J, (state["x"], state["v"]))
        out = dict(J=J.detach(), gx=gx, gv=gv)
        if case["options"] & PARAMS:
            out["params"] = torch.tensor(sim.adjoint_param_gradient(), dtype=torch.float64)
        return out
    if case["kind"] == "host":
        x, v, xo, vo = state["pinned"]
        sim.load(x, v)
        sim.step(case["steps"])
        records = sim.diagnostics()
        capi.pic_get_particles(sim.handle, xo.data_ptr(), vo.data_ptr(), False)
        table = [[r["Wx"], r["Wy"], r["Wz"], r["Q"], r["mode"].real, r["mode"].imag, r["K"]] for r in records]
        return dict(x=xo, v=vo, records=torch.tensor(table, dtype=torch.float64))
    if case["kind"] == "split":
        state["stepper"].step(case["steps"])
    else:
        sim.step(case["steps"])
    x, v = sim.particles(device=True)
    rho, E = _fields(sim)
    return dict(x=x, v=v, rho=rho, E=E)


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    """Per step, each particle's 28 bytes of state are read and written and the field (12 bytes a node) and the
    density (4) cross between grid and particles once; then the results are read and written once.  A reverse step
    reads the 16 bytes of position and moves the 24 bytes of multipliers twice.  Arithmetic, per particle and step:
    about 150 operations (eight corners gathered in three components, rotated, deposited)."""
    s = case["steps"]
    if case["kind"] == "ensemble":
        m = _members(case)
        n, ng = sum(c for _, c, _ in m), sum(a ** 3 for a, _, _ in m)
        return dict(bytes=s * (56 * n + 32 * ng) + 76 * n, flops=150.0 * s * n)
    n, ng = case["particles"], case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "adjoint":
        return dict(bytes=48 * n + s * (56 * n + 32 * ng) + s * (64 * n + 32 * ng) + 72 * n, flops=400.0 * s * n)
    if case["options"] & MOVE:
        return dict(bytes=s * (36 * n + 32 * ng) + 76 * n + 40 * ng, flops=80.0 * s * n)
    total = s * (56 * n + 32 * ng) + 76 * n + 40 * ng
    if case["kind"] == "host":
        total += 48 * n + 28 * n - 40 * ng
    return dict(bytes=total, flops=150.0 * s * n)


def tolerance(case):
    """Measured against `exact` on a GB300: states, densities and fields up to 2.4e-6 (FP32 storage over up to 20
    steps); gradients up to 2.8e-4 on the bump-on-tail sweep, whose per-particle gradients are small beside the
    accumulation's fixed-point unit, and 3e-6 elsewhere."""
    return {"rel": 1.2e-3 if case["kind"] == "adjoint" else 1e-5}


# ------------------------------------------------------------------ the same in 64 bits

def _kvec(n, L, dev):
    k = torch.fft.fftfreq(n, d=1.0 / n, dtype=torch.float64, device=dev)
    g = k.clone()
    if n % 2 == 0:
        g[n // 2] = 0.0
    return 2 * math.pi / L * k, 2 * math.pi / L * g


def _solve(rho, L):
    """E (nz, ny, nx, 3) of a density (nz, ny, nx): -i k_d / |k|^2, no mean, no Nyquist gradient."""
    nz, ny, nx = rho.shape
    kz, gz = _kvec(nz, L, rho.device)
    ky, gy = _kvec(ny, L, rho.device)
    kx, gx = _kvec(nx, L, rho.device)
    k2 = kz[:, None, None] ** 2 + ky[None, :, None] ** 2 + kx[None, None, :] ** 2
    k2[0, 0, 0] = 1.0
    phi = torch.fft.fftn(rho) / k2
    keep = torch.ones_like(k2)
    keep[0, 0, 0] = 0.0
    phi = phi * keep
    g = (gx[None, None, :], gy[None, :, None], gz[:, None, None])
    return torch.stack([torch.fft.ifftn(-1j * g[d] * phi).real for d in range(3)], dim=-1)


def _stencil(y, grid, L):
    """Flat node indices and weights of the eight corners (n, 8); the base is a constant for gradients."""
    n = torch.tensor(grid, dtype=torch.int64, device=y.device)
    s = y / L * n - 0.5
    base = torch.floor(s.detach())
    f = s - base
    base = torch.remainder(base.to(torch.int64), n)
    up = torch.remainder(base + 1, n)
    nodes, weights = [], []
    for c in range(8):
        at = [(up if c >> d & 1 else base)[:, d] for d in range(3)]
        w = [(f if c >> d & 1 else 1 - f)[:, d] for d in range(3)]
        nodes.append(at[0] + grid[0] * (at[1] + grid[1] * at[2]))
        weights.append(w[0] * w[1] * w[2])
    return torch.stack(nodes, 1), torch.stack(weights, 1)


CHUNK = 1 << 22


def _deposit(y, grid, L, q):
    rho = torch.zeros(grid[0] * grid[1] * grid[2], dtype=torch.float64, device=y.device)
    for o in range(0, y.shape[0], CHUNK):
        nodes, w = _stencil(y[o:o + CHUNK], grid, L)
        rho = rho.index_add(0, nodes.reshape(-1), w.reshape(-1))
    dV = L ** 3 / (grid[0] * grid[1] * grid[2])
    return (rho * (q / dV)).reshape(grid[2], grid[1], grid[0])


def _push(y, v, E, grid, L, dt, B, wz2):
    """(y, v) after the kick and the full drift; positions are wrapped only for the quadrupole."""
    ys, vs = [], []
    flat = E.reshape(-1, 3)
    for o in range(0, y.shape[0], CHUNK):
        yc, vc = y[o:o + CHUNK], v[o:o + CHUNK]
        nodes, w = _stencil(yc, grid, L)
        e = (flat[nodes] * w[:, :, None]).sum(1)
        r = yc - (L * torch.floor(yc / L)).detach() - 0.5 * L
        e = e + wz2 * torch.stack([-0.5 * r[:, 0], -0.5 * r[:, 1], r[:, 2]], 1)
        half = -0.5 * dt        # q/m = -1
        m = vc + half * e
        t = (half * B).expand_as(m)
        p = m + torch.linalg.cross(m, t)
        m = m + torch.linalg.cross(p, 2 * t / (1 + (t * t).sum(1, keepdim=True)))
        m = m + half * e
        vs.append(m)
        ys.append(yc + dt * m)
    return torch.cat(ys), torch.cat(vs)


def _wrap(x, L):
    x = torch.remainder(x, L)
    return torch.where(x >= L, x - L, x)


def _splitmix(seed, c):
    """Outputs c of the SplitMix64 generator, as int64 bit patterns."""
    def shift(z, s):
        return (z >> s) & ((1 << (64 - s)) - 1)

    def signed(u):
        return u - (1 << 64) if u >= 1 << 63 else u

    z = signed(seed % (1 << 64)) + c * signed(0x9E3779B97F4A7C15)
    z = (z ^ shift(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ shift(z, 27)) * signed(0x94D049BB133111EB)
    return z ^ shift(z, 31)


def _move(y, step, seed, grid, L):
    pid = torch.arange(y.shape[0], dtype=torch.int64, device=y.device)
    out = torch.empty_like(y)
    for d in range(3):
        r = _splitmix(seed, ((step << 32) + pid) * 4 + d + 1)
        u = ((r >> 40) & 0xFFFFFF).to(torch.float64) / (1 << 24)
        out[:, d] = y[:, d] + (2 * u - 1) * (L / grid[d])
    return out


def _sweep(x, v, grid, family, dt, steps, B, wz2, seed=0, options=0, records=None, mode=None):
    """(y, v, rho, E, used) after `steps` steps from synchronised (x, v): rho of the last positions, E of the last
    solve and the density that it solved for."""
    L, q = FAMILY[family]["L"], _charge(family) / max(1, x.shape[0])
    dV = L ** 3 / (grid[0] * grid[1] * grid[2])
    y = x + 0.5 * dt * v
    E = used = None
    rho = _deposit(y, grid, L, q)
    for s in range(steps):
        used = rho
        E = _solve(rho, L)
        if records is not None:
            at, comp = mode
            F = torch.fft.fftn(E[..., comp])[at[2], at[1], at[0]] / (grid[0] * grid[1] * grid[2])
            W = (E * E).sum(dim=(0, 1, 2)) * dV
            row = [float(W[0]), float(W[1]), float(W[2]), float(rho.sum() * dV), float(F.real), float(F.imag)]
        if options & MOVE:
            y = _move(y, s, seed, grid, L)
        else:
            y, v = _push(y, v, E, grid, L, dt, B, wz2)
        if records is not None:
            records.append(row + [float((v * v).sum() * (-0.5 * q))])     # m_p = q_p / (q/m)
        rho = _deposit(y, grid, L, q)
    return y, v, rho, E, used


def exact(case, seed):
    gen = _gen(seed)
    f = FAMILY[case["family"]]
    L, dev = f["L"], _device()
    B = torch.tensor(f["B"], dtype=torch.float64, device=dev)
    wz2 = torch.tensor(f["wz2"], dtype=torch.float64, device=dev)
    if case["kind"] == "ensemble":
        xs, vs = [], []
        for n, count, alpha in _members(case):
            x, v = _phase_space("landau", count, gen, alpha)
            y, v, _, _, _ = _sweep(x, v, (n,) * 3, "landau", 0.05, case["steps"], B, wz2)
            xs.append(_wrap(y - 0.025 * v, L))
            vs.append(v)
        return dict(x=torch.cat(xs), v=torch.cat(vs))
    grid, dt, N = (case["nx"], case["ny"], case["nz"]), case["dt"], case["particles"]
    if N * case["steps"] > 6e8:     # beyond about 20 seconds
        return None
    x, v = _phase_space(case["family"], N, gen)
    if case["kind"] == "adjoint":
        return _exact_gradient(case, x, v, grid, L, dt, B, wz2)
    mode = (_mode(case)["mode"], _mode(case)["mode_comp"])
    records = [] if case["kind"] == "host" and case["diag_every"] else None
    y, v, rho, E, used = _sweep(x, v, grid, case["family"], dt, case["steps"], B, wz2, int(seed), case["options"],
                                records, mode)
    x = _wrap(y - 0.5 * dt * v, L)
    if case["kind"] == "host":
        return dict(x=x, v=v, records=torch.tensor(records or [], dtype=torch.float64))
    E4 = torch.cat([E, torch.zeros_like(E[..., :1])], dim=-1)
    # a split cycle ends with its push: the density is still the one that was solved for
    return dict(x=x, v=v, rho=used if case["kind"] == "split" else rho, E=E4)


def _exact_gradient(case, x, v, grid, L, dt, B, wz2):
    """J and its gradients by autograd, one step's graph at a time."""
    q = _charge(case["family"]) / x.shape[0]
    dV = L ** 3 / (grid[0] * grid[1] * grid[2])
    leaves = [t.clone().requires_grad_() for t in (x, v, B, wz2)]

    def one(y, v, B, wz2):
        E = _solve(_deposit(y, grid, L, q), L)
        return _push(y, v, E, grid, L, dt, B, wz2)

    y, u = leaves[0] + 0.5 * dt * leaves[1], leaves[1]
    for _ in range(case["steps"] - 1):
        y, u = torch.utils.checkpoint.checkpoint(one, y, u, leaves[2], leaves[3], use_reentrant=False)
    E = _solve(_deposit(y, grid, L, q), L)
    J = (E * E).sum() * dV
    gx, gv, gB, gw = torch.autograd.grad(J, leaves, allow_unused=True)
    out = dict(J=J.detach(), gx=gx, gv=torch.zeros_like(v) if gv is None else gv)
    if case["options"] & PARAMS:
        zero = torch.zeros(3, dtype=torch.float64, device=x.device)
        gB = zero if gB is None else gB
        gw = zero[0] if gw is None else gw
        out["params"] = torch.cat([gB, gw.reshape(1)]).cpu()
    return out

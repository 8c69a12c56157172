"""Readback in load order (GPU): particles that stream freely (no charge) come
back at x0 + n dt v0 with their own velocities, to every kind of destination.

The store holds FP32 offsets and velocities.  Velocities must come back as the
rounded inputs exactly (zeros and subnormals included); a position carries a
rounding of its offset per step, at most 2^-24 cells each, and the FP32 product
dt v, so 1e-6 cells per step plus 1e-6 covers it at |dt v| < 1 cell.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2205_11052_gb300 import capi  # noqa: E402
from paper_2205_11052_gb300.batch import Ensemble  # noqa: E402
from paper_2205_11052_gb300.build import build  # noqa: E402
from paper_2205_11052_gb300.sim import Simulation  # noqa: E402

build()

DT, STEPS = 0.05, 3


def _particles(n, N, L, seed):
    r = np.random.default_rng(seed)
    x, v = r.random((N, 3)) * L, r.standard_normal((N, 3))
    v[:: 7] = 0.0
    v[3:: 11, 1] = 1e-40
    v[5:: 13, 2] = -0.0
    x[0] = 0.0
    if N > 1:
        x[1] = np.nextafter(L, 0.0)
    return x, v


def _check(x, v, x0, v0, n, L):
    v32 = v0.astype(np.float32).astype(np.float64)
    assert np.array_equal(v, v32)
    d = x - (x0 + STEPS * DT * v0)
    d -= L * np.round(d / L)
    assert np.max(np.abs(d) / (np.asarray(L) / np.asarray(n))) < 1e-6 * (STEPS + 1)
    assert x.min() >= 0.0 and np.all(x < L)


@pytest.mark.parametrize("N", [1, 31, 255, 256, 257, 4099, 70_001])
def test_single_run(N):
    n, L = (12, 9, 20), np.array([3.0, 2.5, 4.0])
    x0, v0 = _particles(n, N, L, N)
    sim = Simulation(n=n, L=L, n_particles=N + 5, dt=DT, Q=0.0, sort_period=2, options=1)
    sim.load(x0, v0)
    sim.step(STEPS)
    x, v = sim.particles()
    _check(x, v, x0, v0, n, L)
    xd, vd = sim.particles(device=True)
    assert np.array_equal(xd.cpu().numpy(), x) and np.array_equal(vd.cpu().numpy(), v)
    xp, vp = (torch.empty((N, 3), dtype=torch.float64).pin_memory() for _ in range(2))
    capi.pic_get_particles(sim.handle, xp.data_ptr(), vp.data_ptr(), False)
    assert np.array_equal(xp.numpy(), x) and np.array_equal(vp.numpy(), v)
    sim.step(1)       # the run goes on unharmed by the scratch the readback used
    sim.step(1)
    assert np.array_equal(sim.particles()[1], v)
    sim.close()


def test_ensemble_orders():
    ns, Ns = [(16, 16, 16), (8, 9, 10), (16, 16, 16), (8, 9, 10), (24, 8, 12)], [300, 1, 4097, 0, 255]
    L = np.array([3.0, 2.5, 4.0])
    parts = [_particles(n, N, L, 50 + i) if N else (np.zeros((0, 3)), np.zeros((0, 3)))
             for i, (n, N) in enumerate(zip(ns, Ns))]
    ens = Ensemble([(n, L, x, v, 0.0) for n, (x, v) in zip(ns, parts)], dt=DT, sort_period=2, options=1)
    ens.step(STEPS)
    xs, vs = ens.particles()
    for (x0, v0), x, v, n in zip(parts, xs, vs, ns):
        if x0.size:
            _check(x, v, x0, v0, n, L)
    N = sum(Ns)
    xd, vd = (torch.empty((N, 3), dtype=torch.float64, device="cuda") for _ in range(2))
    capi.pic_batch_get_particles(ens.handle, xd.data_ptr(), vd.data_ptr(), True)
    assert np.array_equal(xd.cpu().numpy(), np.concatenate(xs))
    assert np.array_equal(vd.cpu().numpy(), np.concatenate(vs))
    ens.close()


@pytest.mark.parametrize("copies", [1, 40])
def test_ensemble_offsets_come_back_exactly(copies):
    """Unit spacing: node + offset is exact in FP64 for offsets down to 2^-42, around
    2^-19 (where the sum changes from integer to FP64 instructions) and up to 1."""
    off = np.array([0.0, 2.0**-42, 2.0**-20 * (2 - 2.0**-23), 2.0**-19, 2.0**-19 * (1 + 2.0**-23), 0.5,
                    1 - 2.0**-24])
    sizes = [(24, 16, 9), (1000, 8, 8), (24, 16, 9)]
    r = np.random.default_rng(9)
    insts = []
    for n in sizes:
        i = np.tile(np.arange(n[0]), copies)
        idx = np.stack([i, r.integers(0, n[1], i.size), r.integers(0, n[2], i.size)], 1)
        x = idx + 0.5 + off[r.integers(0, off.size, idx.shape)]
        insts.append((n, np.array(n, dtype=float), x, np.zeros_like(x), 0.0))
    ens = Ensemble(insts, dt=DT)
    xs, vs = ens.particles()
    for (n, L, x0, v0, _), x, v in zip(insts, xs, vs):
        assert np.array_equal(x, np.mod(x0, L)) and np.array_equal(v, v0)
    ens.close()


@pytest.mark.parametrize("shift", [0, -1, 1, 37, -2**20, 2**30])
def test_positions_load_exactly(shift):
    """Unit spacing: nodes plus offsets that FP32 and FP64 both hold, whole boxes away,
    the first half cell (below node 0) and offsets around 2^-26 included, where the
    load goes from integer to FP64 instructions."""
    n = (24, 16, 9)
    L = np.array(n, dtype=float)
    tiny = 2.0**-40 if abs(shift) < 2 else 2.0**-12
    off = np.array([0.0, tiny, 2.0**-26, 2.0**-27, 2.0**-26 * (1 + 2.0**-10), 0.25, 0.5, 1 - 2.0**-12])
    off = off[off >= tiny] if abs(shift) >= 2 else off
    r = np.random.default_rng(3)
    N = 5000
    idx = np.stack([r.integers(0, m, N) for m in n], 1)
    x = idx + 0.5 + off[r.integers(0, off.size, idx.shape)] + shift * L
    x[:10] = [[0.25, 0.5 - 2.0**-20, 2.0**-10]] * 10 + shift * L     # below node 0
    v = r.standard_normal((N, 3)) * 10.0 ** r.integers(-42, 30, (N, 3))
    sim = Simulation(n=n, L=L, n_particles=N, dt=0.0 + 1e-300, Q=0.0)
    sim.load(x, v)
    xg, vg = sim.particles()
    v32 = v.astype(np.float32).astype(np.float64)
    assert np.array_equal(vg, v32)
    assert np.array_equal(xg, np.mod(x, L))
    sim.close()

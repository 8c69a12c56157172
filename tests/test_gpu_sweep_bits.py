"""The forward sweep of a gradient keeps its bits (needs a GPU).

The derivative of the cloud-in-cell weights jumps where a particle crosses a cell
face, and the last step's deposit enters the gradient without a factor dt.  So a
particle within rounding of a face at the last step has a gradient that hangs on
the last bits of the trajectory, and a sweep whose field solve is rounded otherwise
gives another one, by up to a tenth of the largest component.  The sweeps therefore
go through the same transforms on every grid: their states are pinned bit for bit,
on grids where runs use the library's own transforms, and away from the faces the
gradient is held to the oracle's.

The pinned checksums (tests/golden/gradient_sweep_bits.json) come from the library
before it had transforms of its own; `python tests/test_gpu_sweep_bits.py` prints
those of the present one.  They hold for cuFFT of CUDA 13.0: another release may
round otherwise.
"""
import json
import os
import sys
import zlib

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if __name__ == "__main__":
    sys.path.insert(0, sys.argv[1] if len(sys.argv) > 1 else ROOT)

import pic_inputs as pi
from oracle import pic_oracle as po

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2205_11052_gb300 import capi  # noqa: E402
from paper_2205_11052_gb300.build import build  # noqa: E402
from paper_2205_11052_gb300.sim import Simulation  # noqa: E402

pytestmark = pytest.mark.gpu

build()

GOLDEN = os.path.join(ROOT, "tests", "golden", "gradient_sweep_bits.json")
FIXED = capi.PIC_OPT_FIXED_DEPOSIT
# name: (grid, particles, B, wz2, settings); 24^3 and 8^3 are grids on which cuFFT's
# planar and interleaved transforms differ in bits
CASES = {
    "64": ((64, 64, 64), 400_000, (0.0, 0.0, 0.0), 0.0, {}),
    "24_trap": ((24, 24, 24), 60_001, (0.0, 0.0, 5.0), 1.0, dict(guard=3)),
    "ragged": ((45, 28, 36), 100_007, (0.1, 0.2, 0.3), 0.5, dict(sort_period=2)),
    "8": ((8, 8, 8), 4_000, (0.0, 0.0, 0.0), 0.0, {}),
    "flat": ((96, 48, 2), 30_000, (0.0, 0.0, 0.0), 0.0, dict(tile=(4, 4, 2))),
    "primes": ((37, 41, 29), 90_001, (0.0, 0.0, 0.0), 0.0, {}),
}
L = 62.5


def _inputs(n):
    """Made of sums and products alone, so that every machine draws the same bits."""
    rng = np.random.default_rng(77)
    u = rng.random((n, 3))
    x = L * (u - 0.15 * u * (1.0 - u))
    v = rng.random((n, 3, 6)).sum(axis=2) - 3.0
    return x, v


def _checksums(name):
    grid, n, B, wz2, kw = CASES[name]
    sim = Simulation(n=grid, L=(L,) * 3, n_particles=n, dt=0.05, Q=-L ** 3, B=B, wz2=wz2, options=FIXED, **kw)
    sim.load(*_inputs(n))
    sim.adjoint_forward(8, checkpoint_every=3)
    v = sim.particles()[1].astype(np.float32)      # as stored
    rho, E = sim.field()
    rho = rho + np.float32(0.0)                    # an empty node's zero has no sign
    assert sim.flags() == 0
    sim.close()
    return {k: zlib.crc32(np.ascontiguousarray(a).tobytes()) for k, a in (("v", v), ("rho", rho), ("E", E))}


@pytest.mark.parametrize("name", list(CASES))
def test_the_forward_sweep_keeps_its_bits(name):
    with open(GOLDEN) as f:
        assert _checksums(name) == json.load(f)[name]


def test_recomputed_segments_repeat_the_forward_sweep():
    """Gradients with recomputed segments and with every step kept come from the
    same trajectory; what is left is the order of the reverse deposits' FP32 adds."""
    grid, n, B, wz2, kw = CASES["24_trap"]
    sim = Simulation(n=grid, L=(L,) * 3, n_particles=n, dt=0.05, Q=-L ** 3, B=B, wz2=wz2, options=FIXED, **kw)
    sim.load(*_inputs(n))
    out = []
    for keep in (8, 2):
        sim.adjoint_forward(8, checkpoint_every=keep)
        out.append(sim.adjoint_backward())
    sim.close()
    for a, b in zip(*out):
        assert np.max(np.abs(a - b)) <= 1e-5 * np.max(np.abs(a))


@pytest.mark.parametrize("name", ["24_trap", "primes"])
@pytest.mark.parametrize("steps,keep,last", [(8, 3, 3), (8, 8, 8), (5, 2, 2), (1, 4, 1)])
def test_fields_after_a_gradient_are_the_last_ones(name, steps, keep, last):
    """Segments are recomputed back to front, so the last solve is that of the first
    segment's last step and the last deposit that of its push (or both are the
    objective's where nothing is recomputed)."""
    grid, n, B, wz2, kw = CASES[name]
    rho, E = [], []
    for s, k, back in ((steps, keep, True), (last, last, False), (last + (last < steps), last + 1, False)):
        sim = Simulation(n=grid, L=(L,) * 3, n_particles=n, dt=0.05, Q=-L ** 3, B=B, wz2=wz2, options=FIXED, **kw)
        sim.load(*_inputs(n))
        sim.adjoint_forward(s, checkpoint_every=k)
        if back:
            sim.adjoint_backward()
        f = sim.field()
        rho.append(f[0])
        E.append(f[1])
        sim.close()
    assert np.array_equal(E[0], E[1])
    assert np.array_equal(rho[0], rho[2])


def test_gradient_away_from_cell_faces():
    """Particles farther than 1e-4 cells (a hundred times the FP32 trajectory's error)
    from a face at the last step: 2-norm of the difference to the oracle within 1e-5
    of the gradient's, the FP32 field's error (2e-7 of E, amplified by the derivative
    of a field that varies over many cells)."""
    w = pi.bump_on_tail(n=24, ppc=16, seed=31, alpha=0.05, k=0.1)
    steps = 12
    sim = Simulation.from_workload(w, options=FIXED, sort_period=4)
    J = sim.adjoint_forward(steps, (1.0, 1.0, 1.0), checkpoint_every=4)
    gx, gv = sim.adjoint_backward()
    sim.close()
    g = po.Grid(w.n, w.L)
    p = po.Params(dt=w.dt, Q=w.Q, q_over_m=w.q_over_m)
    Jo, gxo, gvo = po.run_with_gradient(w.x, w.v, g, p, steps, (1.0, 1.0, 1.0))
    x, v, _ = po.run(w.x, w.v, g, p, steps - 1)
    s = (x + 0.5 * w.dt * v) / (np.asarray(w.L) / np.asarray(w.n)) - 0.5
    away = np.all(np.abs(s - np.round(s)) > 1e-4, axis=1)
    assert 0.9 < away.mean() < 1.0
    assert J == pytest.approx(Jo, rel=1e-5)
    for got, ref in ((gx, gxo), (gv, gvo)):
        assert np.linalg.norm((got - ref)[away]) <= 1e-5 * np.linalg.norm(ref[away])


if __name__ == "__main__":
    print(json.dumps({name: _checksums(name) for name in CASES}, indent=1))

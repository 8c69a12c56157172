"""The fused push reads E along three paths that must give the same bits
(needs a GPU).

`k_push_deposit` gathers E (Section 3.1 step 3) from a shared-memory copy of
its tile's box when that copy fits two blocks per SM, with the box extent
compiled in for 8^3 tiles with two guard layers, and with three (whose box has
two); particles outside the box, and every particle when the copy does not fit
with two layers, read the x-paired grid. All
paths read the same E values and interpolate them in the same order, and the
fixed-point deposit sums integers, so a run gives bit-identical particles and
charge density whichever path each particle takes. Without re-binning after
the load, particles drift out of their tiles' boxes, so the grid path runs
beside the shared one within a launch.
"""
import numpy as np
import pytest

import pic_inputs as pi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2205_11052_gb300 import capi  # noqa: E402
from paper_2205_11052_gb300.build import build  # noqa: E402
from paper_2205_11052_gb300.sim import Simulation  # noqa: E402

build()

# (tile, guard): the staged box with the compiled-in extent (13 slots per
# axis), a staged box of another shape (13 x 13 x 11 slots), the staged box with
# fewer layers than the deposit's, and a deposit tile (19^3 slots) beside which not
# even two layers fit (E from the grid)
PATHS = {
    "staged_constant_box": ((8, 8, 8), 2),
    "staged_runtime_box": ((8, 8, 6), 2),
    "staged_fewer_layers": ((8, 8, 8), 3),
    "grid_only": ((8, 8, 8), 5),
}


def _run(w, tile, guard, steps=6):
    sim = Simulation.from_workload(w, tile=tile, guard=guard, sort_period=-1,
                                   options=capi.PIC_OPT_FIXED_DEPOSIT)
    sim.step(steps)
    x, v = sim.particles()
    rho, _ = sim.field()
    _, strays = sim.rebin_stats()
    flags = sim.flags()
    sim.close()
    return x, v, rho, strays, flags


def test_staged_and_grid_gathers_give_the_same_bits():
    # dt = 0.3 moves a thermal particle about 0.8 cells per step on this grid
    w = pi.landau(n=32, ppc=8, alpha=0.2, seed=21, dt=0.3)
    runs = {name: _run(w, *cfg) for name, cfg in PATHS.items()}
    ref = runs["staged_constant_box"]
    assert ref[4] == 0
    # particles left their boxes, so both gather paths and the stray deposit ran
    assert ref[3] > w.n_particles // 100
    for name, got in runs.items():
        assert got[4] == 0, name
        for a, b, what in zip(ref[:3], got[:3], ("x", "v", "rho")):
            assert np.array_equal(a, b), f"{name}: {what} differs"


@pytest.mark.parametrize("tile,guard", list(PATHS.values()), ids=list(PATHS))
@pytest.mark.parametrize("kw", [{}, dict(B=(0.1, -0.2, 5.0), wz2=1.0)], ids=["plain", "trap"])
def test_split_calls_and_steps_give_the_same_bits(tile, guard, kw):
    """deposit, solve and gather + push called one by one do what a step does."""
    w = pi.landau(n=32, ppc=8, alpha=0.2, seed=22, dt=0.3)
    out = []
    for split in (False, True):
        sim = Simulation.from_workload(w, tile=tile, guard=guard, sort_period=-1,
                                       options=capi.PIC_OPT_FIXED_DEPOSIT, **kw)
        for _ in range(4):
            if split:
                sim.deposit()
                sim.field_solve()
                sim.gather_push()
            else:
                sim.step(1)
        if split:
            sim.deposit()
        out.append((*sim.particles(), sim.field()[0]))
        assert sim.flags() == 0
        sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)

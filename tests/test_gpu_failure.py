"""Failure detection without a GPU fault (needs a GPU).

The staged kernels wait for their bulk copies on mbarriers with a bounded
wait.  pic_selftest_timeout runs one such wait with nothing to wait for: it
must give up within its limit, raise PIC_FLAG_TIMEOUT, report
PIC_ERR_TIMEOUT, and leave the context usable.  Nothing here faults, traps or
hangs the GPU: the wait is bounded in time and no copy is in flight.
"""
import time

import numpy as np
import pytest

import pic_inputs as pi
from oracle import pic_oracle as po

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2205_11052_gb300 import capi  # noqa: E402
from paper_2205_11052_gb300.build import build  # noqa: E402
from paper_2205_11052_gb300.sim import Simulation  # noqa: E402

build()


def test_a_bounded_wait_that_runs_out_is_reported_and_the_context_survives():
    w = pi.landau(n=16, ppc=8, seed=51)
    sim = Simulation.from_workload(w, diag_every=1)
    t0 = time.perf_counter()
    rc = capi.pic_selftest_timeout(sim.handle)
    secs = time.perf_counter() - t0
    assert rc == capi.PIC_ERR_TIMEOUT
    assert secs < 30.0
    assert sim.flags() & capi.PIC_FLAG_TIMEOUT
    sim.step(1)
    with pytest.raises(capi.PicError) as e:
        sim.diagnostics()
    assert e.value.code == capi.PIC_ERR_TIMEOUT
    # cleared, the same context runs on and matches the oracle
    assert sim.flags(clear=True) & capi.PIC_FLAG_TIMEOUT
    assert sim.flags() == 0
    sim.step(2)
    x, v = sim.particles()
    hist = sim.diagnostics()
    sim.close()
    assert len(hist) == 3
    xo, vo, _ = po.run(w.x, w.v, po.Grid(w.n, w.L), po.Params(dt=w.dt, Q=w.Q), 3)
    L = np.asarray(w.L)
    d = x - xo
    d -= L * np.round(d / L)
    assert np.max(np.abs(d) / (L / np.asarray(w.n))) <= 1e-4
    assert np.max(np.abs(v - vo)) <= 1e-4 * np.max(np.abs(vo))


def _load_indices(sim):
    """int32 views of the arena's load-index arrays: the 256-byte aligned places that hold
    a permutation of the particles."""
    n = sim.n_particles
    total, squares = n * (n - 1) // 2, (n - 1) * n * (2 * n - 1) // 6
    words = sim.arena.view(torch.int32)
    found = []
    for off in range(0, words.numel() - n + 1, 64):
        a = words[off:off + n]
        if 0 <= int(a[0]) < n and 0 <= int(a[-1]) < n and int(a.min()) >= 0 and int(a.max()) < n:
            b = a.to(torch.int64)
            if int(b.sum()) == total and int((b * b).sum()) == squares:
                found.append(a)
    return found


def test_load_indices_of_a_binning_that_gave_up_are_not_followed():
    """A re-binning that gives up leaves slots with other bits in the place of load
    indices.  The arena is put into that state: the readback and the gradient finish, and
    every particle that still has its index comes back as without.  (Its gradient does
    not: the multipliers of the lost ones are missing in the adjoint fields.)"""
    w = pi.bump_on_tail(n=8, ppc=4, seed=52, alpha=0.2, k=0.5)
    out = []
    for broken in (False, True):
        sim = Simulation.from_workload(w, sort_period=2, options=capi.PIC_OPT_FIXED_DEPOSIT)
        sim.sort()
        sim.stream.synchronize()
        if broken:
            arrays = _load_indices(sim)
            assert arrays
            lost = torch.unique(torch.cat([a[100:140] for a in arrays])).cpu().numpy()
            for a in arrays:
                a[100:120] = 0x3F800000       # 1.0f
                a[120:140] = -0x40800000      # -1.0f
        x, v = sim.particles()
        xd, vd = sim.particles(device=True)
        J = sim.adjoint_forward(7, checkpoint_every=3)
        gx, gv = sim.adjoint_backward()
        out.append((x, v, xd.cpu().numpy(), vd.cpu().numpy(), gx, gv, J))
        sim.close()
    keep = np.setdiff1d(np.arange(w.n_particles), lost)
    assert len(keep) >= w.n_particles - 80
    ref, got = out
    for a, b in zip(ref[:4], got[:4]):
        assert np.array_equal(a[keep], b[keep])
    for a in got[4:6]:
        assert np.all(np.isfinite(a[keep]))
    assert got[6] == ref[6]

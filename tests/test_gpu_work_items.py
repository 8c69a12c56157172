"""Work items, folds and staged boxes at their edges (GPU).

Particle counts around the block, item and fold sizes, single tiles that one block
cannot take without folding, grids of more tiles than a sort's last block walks, and
the reverse push with and without staged boxes, each against the oracle at the
parity tests' tolerances (FP32 against FP64: 1e-5 of the largest value, gradients
1e-4).
"""
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

FIXED = capi.PIC_OPT_FIXED_DEPOSIT


def _check_steps(n, L, N, options, seed, steps=2, **kw):
    """rho of the start and the state after some fused steps."""
    r = np.random.default_rng(seed)
    x, v = r.random((N, 3)) * np.asarray(L), r.standard_normal((N, 3))
    Q = -float(np.prod(L))
    sim = Simulation(n=n, L=L, n_particles=N, dt=0.02, Q=Q, options=options, **kw)
    sim.load(x, v)
    sim.deposit()
    rho, _ = sim.field()
    g = po.Grid(n, L)
    want = po.deposit(po.wrap(x + 0.01 * v, g), g, Q / N)
    assert np.max(np.abs(rho - want)) <= 1e-5 * np.max(np.abs(want))
    sim.step(steps)
    xg, vg = sim.particles()
    xo, vo, _ = po.run(x, v, g, po.Params(dt=0.02, Q=Q), steps, diag_every=0)
    d = xg - xo
    d -= np.asarray(L) * np.round(d / np.asarray(L))
    assert np.max(np.abs(d) / g.h) <= 1e-5 * steps
    assert np.max(np.abs(vg - vo)) <= 1e-5 * steps * np.max(np.abs(vo))
    assert sim.flags() == 0
    sim.close()


@pytest.mark.parametrize("options", [0, FIXED], ids=["fp32", "fixed"])
@pytest.mark.parametrize("N", [63, 64, 255, 257, 384, 385, 1000, 3839, 3841, 7681, 60_000])
def test_counts_around_block_and_item_sizes(N, options):
    _check_steps((8, 8, 8), (1.0, 1.2, 0.9), N, options, N)
    _check_steps((20, 9, 12), (3.0, 1.2, 2.0), N, options, N + 1, tile=(4, 4, 4), guard=1, sort_period=2)


@pytest.mark.parametrize("options", [0, FIXED], ids=["fp32", "fixed"])
def test_one_tile_with_more_particles_than_a_fold(options):
    _check_steps((8, 8, 8), (1.0, 1.2, 0.9), 3_000_001, options, 1, steps=1)


@pytest.mark.parametrize("chunk", [32, 100, 4095])
def test_items_of_the_callers_size(chunk):
    _check_steps((16, 16, 16), (2.0, 2.0, 2.0), 30_011, FIXED, chunk, chunk=chunk)


def test_more_tiles_than_the_fused_passes_take():
    """33^3 = 35937 tiles: the sort's separate kernels, bit for bit against the run
    that never re-bins (the fixed-point deposit does not depend on the order)."""
    n, L, N = (132, 132, 132), (4.0, 4.0, 4.0), 200_003
    r = np.random.default_rng(3)
    x, v = r.random((N, 3)) * 4.0, r.standard_normal((N, 3))
    out = []
    for period in (1, -1):
        sim = Simulation(n=n, L=L, n_particles=N, dt=0.01, Q=-64.0, options=FIXED, tile=(4, 4, 4),
                         sort_period=period)
        sim.load(x, v)
        sim.step(3)
        out.append(sim.particles())
        sim.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


# 21^3 = 9261 tiles, 37 KB of counters; 24^3 = 13824 and 32^3 = 32768, 55 and 131 KB, above
# what a block has without asking; each with enough particles (four times the tiles for
# each of 152 blocks) for counters in shared memory
@pytest.mark.parametrize("axis,N", [(84, 6_000_001), (96, 9_000_001), (128, 20_000_001)])
def test_histogram_of_more_keys_than_small_blocks_take(axis, N):
    assert -(-N // 152) >= 4 * (axis // 4) ** 3
    n, L = (axis,) * 3, (4.0, 4.0, 4.0)
    r = np.random.default_rng(4)
    x, v = r.random((N, 3)) * 4.0, r.standard_normal((N, 3))
    out = []
    for period in (1, -1):
        sim = Simulation(n=n, L=L, n_particles=N, dt=0.01, Q=-64.0, options=FIXED, tile=(4, 4, 4),
                         sort_period=period)
        sim.load(x, v)
        sim.step(2)
        out.append(sim.particles())
        assert sim.flags() == 0
        sim.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


# (tile, guard): field boxes of the deposit's guard layers (2, 1), of fewer (3, 4 and
# an uneven tile) and none at all (5)
BOXES = [((8, 8, 8), 3), ((8, 8, 8), 4), ((8, 8, 8), 5), ((8, 6, 8), 3), ((4, 8, 8), 5), ((4, 4, 4), 1)]


@pytest.mark.parametrize("tile,guard", BOXES)
def test_field_boxes_of_fewer_layers_give_the_same_bits(tile, guard):
    w = pi.landau(n=24, ppc=8, alpha=0.2, seed=22, dt=0.3)   # 0.6 cells a step
    out = []
    for kw in (dict(tile=(8, 8, 8), guard=2), dict(tile=tile, guard=guard)):
        sim = Simulation.from_workload(w, sort_period=-1, options=FIXED, **kw)
        sim.step(6)
        out.append((*sim.particles(), sim.field()[0]))
        assert sim.flags() == 0
        sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("tile,guard", BOXES[:4])
def test_field_boxes_of_fewer_layers_with_fp32_deposit(tile, guard):
    _check_steps((24, 24, 24), (2.0, 2.0, 2.0), 20_011, 0, guard, steps=4, tile=tile, guard=guard,
                 sort_period=-1)


@pytest.mark.parametrize("n", [(17, 9, 25), (41, 41, 41), (64, 64, 8)])
@pytest.mark.parametrize("N", [5000, 174_646, 1_500_001])
def test_shares_of_a_bunch_among_thin_tiles(n, N):
    """Half the particles in a few cells, half anywhere: whatever the items and the
    blocks' shares, the fixed-point deposit gives the same bits."""
    L = np.asarray(n) * 0.1
    r = np.random.default_rng(N)
    x, v = r.random((N, 3)) * L, r.standard_normal((N, 3))
    x[::2] = (0.6 + 0.05 * r.standard_normal((x[::2].shape))) % L
    out = []
    for chunk in (0, 32, 4095):
        sim = Simulation(n=n, L=L, n_particles=N, dt=0.01, Q=-float(np.prod(L)), options=FIXED,
                         sort_period=2, chunk=chunk)
        sim.load(x, v)
        sim.step(3)
        out.append((*sim.particles(), sim.field()[0]))
        assert sim.flags() == 0
        sim.close()
    for o in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(out[0], o))


@pytest.mark.parametrize("kw", [dict(), dict(guard=3), dict(tile=(4, 4, 4), guard=1), dict(guard=8)],
                         ids=["staged", "grid", "small-box", "large-box"])
def test_reverse_push_shapes(kw):
    w = pi.bump_on_tail(n=12, ppc=6, seed=5, alpha=0.2, k=0.5)
    w.dt = 0.1
    weights, steps = (0.0, 0.5, 1.0), 5
    sim = Simulation.from_workload(w, options=FIXED, sort_period=2, **kw)
    J = sim.adjoint_forward(steps, weights, checkpoint_every=3)
    gx, gv = sim.adjoint_backward()
    Jo, gxo, gvo = po.run_with_gradient(w.x, w.v, po.Grid(w.n, w.L),
                                        po.Params(dt=w.dt, Q=w.Q, q_over_m=w.q_over_m), steps, weights)
    assert J == pytest.approx(Jo, rel=1e-5)
    assert np.max(np.abs(gx - gxo)) <= 1e-4 * np.max(np.abs(gxo))
    assert np.max(np.abs(gv - gvo)) <= 1e-4 * np.max(np.abs(gvo))
    sim.close()

"""The density of the fixed-point deposit is the FP64 product of the integer sums
and the scale, rounded once to FP32 (needs a GPU).

Particles at multiples of 1/64 of a cell have weights that are whole multiples of
2^-18, so the deposit's integer sums are known exactly.  The charges are chosen so
that a node's product lies so close to halfway between two floats that a product
carried in FP32 pairs rounds the other way (found by emulating it over 5e4 charges).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2205_11052_gb300 import capi  # noqa: E402
from paper_2205_11052_gb300.build import build  # noqa: E402
from paper_2205_11052_gb300.sim import Simulation  # noqa: E402

build()

N, PARTICLES = 16, 409_601


def _sums():
    """Particles in units of 1/64 cell from the node, and the sums in units of 2^-20."""
    rng = np.random.default_rng(3)
    cell = rng.integers(0, N, (PARTICLES, 3))
    k = rng.integers(0, 64, (PARTICLES, 3))
    cell[:PARTICLES // 2] = cell[:PARTICLES // 2] % 5      # uneven nodes
    q = np.zeros(N ** 3, np.int64)
    for c in range(8):
        w, node = np.ones(PARTICLES, np.int64), np.zeros(PARTICLES, np.int64)
        for d, stride in enumerate((1, N, N * N)):
            up = c >> d & 1
            w *= k[:, d] if up else 64 - k[:, d]
            node += (cell[:, d] + up) % N * stride
        np.add.at(q, node, 4 * w)
    assert q.sum() == PARTICLES << 20
    return cell + 0.5 + k / 64.0, q


# near-halfway charges, then scales at the ends of the FP32 range and a plain one
@pytest.mark.parametrize("Q", [-946.010667, -3814.935696, -867.703632, -971.452847, -392.727415, -133.66836,
                               -1e-30, 1e33, -4096.0])
def test_density_is_the_fp64_product_rounded_once(Q):
    x, q = _sums()
    sim = Simulation(n=(N,) * 3, L=(float(N),) * 3, n_particles=PARTICLES, dt=0.05, Q=Q,
                     options=capi.PIC_OPT_FIXED_DEPOSIT)
    sim.load(x, np.zeros_like(x))
    sim.deposit()
    rho, _ = sim.field()
    sim.close()
    want = (q.astype(np.float64) * (Q / PARTICLES / 1.0 / 1048576.0)).astype(np.float32)
    assert np.array_equal(rho.reshape(-1), want)

"""The field solve on grids that take each of its paths (GPU): the library's own
line transforms (every radix, primes, ragged boxes, short and unit axes), and cuFFT
beyond them; with the records' field sums against the field itself.

Tolerance: an FP32 transform of N points carries about sqrt(log2 N) roundings of
2^-24 in the mean, and the solve has two of them and the products between; 1e-5 of
the largest value is the parity tests' bound.
"""
import numpy as np
import pytest

from oracle import pic_oracle as po

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU-only machines
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2205_11052_gb300 import capi  # noqa: E402
from paper_2205_11052_gb300.build import build  # noqa: E402
from paper_2205_11052_gb300.sim import Simulation  # noqa: E402

build()

GRIDS = [(2, 1, 1), (3, 2, 1), (4, 1, 5), (16, 16, 16), (24, 36, 28), (45, 49, 20), (33, 17, 31),
         (62, 29, 26), (26, 33, 39), (64, 64, 64), (96, 7, 100), (19, 23, 121), (127, 16, 8), (112, 112, 16),
         (128, 128, 12), (130, 24, 9), (8, 74, 12)]


@pytest.mark.parametrize("n", GRIDS, ids=str)
def test_field_of_a_density(n):
    L = (3.0, 2.5, 4.0)
    rho = np.random.default_rng(sum(n)).standard_normal((n[2], n[1], n[0])).astype(np.float32)
    sim = Simulation(n=n, L=L, n_particles=1, dt=0.05, Q=0.0)
    sim.set_rho(rho)
    sim.field_solve()
    got, E = sim.field()
    want = po.solve_field(rho.astype(np.float64), po.Grid(n, L))
    assert np.array_equal(got, rho)
    assert np.max(np.abs(E - want)) <= 1e-5 * max(np.max(np.abs(want)), 1e-30)
    sim.close()


@pytest.mark.parametrize("n", [(16, 16, 16), (45, 49, 20), (130, 24, 9)], ids=str)
def test_sums_and_mode_of_a_record(n):
    L = (3.0, 2.5, 4.0)
    r = np.random.default_rng(7)
    x, v = r.random((5000, 3)) * np.asarray(L), np.zeros((5000, 3))
    sim = Simulation(n=n, L=L, n_particles=5000, dt=1e-3, Q=-2.0, diag_every=1, options=1,
                     mode=(1, 2, -1), mode_comp=1)
    sim.load(x, v)
    sim.deposit()
    rho, _ = sim.field()
    sim.step(1)
    rec = sim.diagnostics()[0]
    _, E = sim.field()
    dV = np.prod(L) / np.prod(n)
    for d, w in enumerate(("Wx", "Wy", "Wz")):
        assert rec[w] == pytest.approx(dV * np.sum(E[d].astype(np.float64) ** 2), rel=1e-9)
    assert rec["Q"] == pytest.approx(dV * np.sum(rho.astype(np.float64)), rel=1e-9)
    m = po.mode_coefficient(E[1].astype(np.float64), (1, 2, -1))
    scale = np.sqrt(np.mean(E[1].astype(np.float64) ** 2))
    assert abs(rec["mode"] - m) <= 1e-5 * scale
    sim.close()


def test_field_sums_of_runs_and_ensembles():
    """Field energies and charge against the exact sums of the same field and density:
    within 4e-16, a few of FP64's roundings (in pairs of FP32 the squares are off by 4e-16
    to 8e-16, their last bits not being random).  A run and an ensemble's instance of one grid have
    the same field."""
    import math

    from paper_2205_11052_gb300.batch import Ensemble

    rng = np.random.default_rng(61)
    L = 12.0
    members = [(n, L, rng.random((N, 3)) * L, rng.standard_normal((N, 3)), -L ** 3)
               for n, N in ((16, 40_000), (32, 500_001), (48, 600_003), (60, 900_000))]
    ens = Ensemble(members, dt=0.01, options=capi.PIC_OPT_FIXED_DEPOSIT, diag_every=1)
    ens.step(1)
    records = ens.diagnostics()[-1]
    ens.close()
    for (n, _, x, v, Q), rec in zip(members, records):
        sim = Simulation(n=(n,) * 3, L=(L,) * 3, n_particles=len(x), dt=0.01, Q=Q, diag_every=1,
                         options=capi.PIC_OPT_FIXED_DEPOSIT)
        sim.load(x, v)
        sim.deposit()
        sim.field_solve()
        rho, E = sim.field()
        sim.step(1)
        own = sim.diagnostics()[-1]
        sim.close()
        dV = (L / n) ** 3
        for key, a in (("Wx", E[0].astype(np.float64) ** 2), ("Wy", E[1].astype(np.float64) ** 2),
                       ("Wz", E[2].astype(np.float64) ** 2), ("Q", rho.astype(np.float64))):
            exact = dV * math.fsum(a.ravel())
            for got in (rec[key], own[key]):
                assert abs(got - exact) <= 4e-16 * abs(exact), (n, key)

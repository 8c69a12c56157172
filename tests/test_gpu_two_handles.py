"""Several runs in one process (needs a GPU): binding one changes nothing for another.

A kernel's limit of dynamic shared memory belongs to the function, not to a handle.
Each pair below binds a run whose tiles take more shared memory, then one that takes
less, and steps them in turn; each must go as it goes alone.
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

FIXED, MOVE = capi.PIC_OPT_FIXED_DEPOSIT, capi.PIC_OPT_UNIFORM_MOVE


def _split(sim):
    sim.deposit()
    sim.field_solve()
    sim.gather_push()


def _gradient(sim):
    sim.adjoint_forward(3, checkpoint_every=2)
    sim._gradient = sim.adjoint_backward()


# what is run, the settings of the run bound first, those of the run bound second
PAIRS = {
    "step": (lambda s: s.step(1), dict(guard=3), dict()),
    "step_fp32": (lambda s: s.step(1), dict(guard=3, options=0), dict(options=0)),
    "move": (lambda s: s.step(1), dict(guard=5, options=FIXED | MOVE), dict(guard=4, options=FIXED | MOVE)),
    "split": (_split, dict(guard=5), dict(guard=4)),
    "gradient": (_gradient, dict(guard=3), dict()),
}


def _make(w, kw):
    return Simulation.from_workload(w, sort_period=2, **dict(dict(options=FIXED), **kw))


def _state(sim):
    out = list(sim.particles())
    if hasattr(sim, "_gradient"):
        out += sim._gradient
    return out


@pytest.mark.parametrize("name", list(PAIRS))
def test_runs_of_different_tiles_do_not_disturb_each_other(name):
    run, first, second = PAIRS[name]
    w = pi.landau(n=16, ppc=8, alpha=0.1, seed=41)
    alone = []
    for kw in (first, second):
        sim = _make(w, kw)
        for _ in range(3):
            run(sim)
        alone.append(_state(sim))
        sim.close()
    sims = [_make(w, first), _make(w, second)]
    for _ in range(3):
        for sim in sims:
            run(sim)
    for sim, ref in zip(sims, alone):
        assert sim.flags() == 0
        for a, b in zip(_state(sim), ref):
            # FP32 adds of the density and the reverse deposit come in any order
            if name in ("step_fp32", "gradient"):
                assert np.max(np.abs(a - b)) <= 1e-5 * np.max(np.abs(b))
            else:
                assert np.array_equal(a, b)
        sim.close()

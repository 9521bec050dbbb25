"""The step kernels' launches: flat ones (the plane's units numbered through,
rows not rounded up to blocks), the small blocks of lattices below one wave and
consecutive steps as programmatic dependent launches give, bit for bit, the
populations of a shaped launch of single-warp blocks, eagerly, in graphs and
after autotuning; the diagnosing step in a flat launch gives the standalone
diagnostics of the same state."""
import numpy as np
import pytest

import stgv_inputs as I
from paper_2605_14505_gb300 import lbm

from _helpers import lattice_params

pytestmark = pytest.mark.gpu


def _sim(shape, pair, forcing, storage):
    nx, ny, nz = shape
    sim = lbm.Simulation(lattice_params(nx, ny, nz, pair, forcing, 0.55, 0.6, 3e-3 / 1024, -3e-3 * 1024),
                         storage=storage)
    sim.init_fields(*I.random_fields(nx, ny, nz, 4, 0.03, 0.01, 0.1))
    return sim


@pytest.mark.parametrize("shape,pair,forcing,storage", [
    ((1, 5, 3), "19x7", "guo", "fp32"),      # rows of one node: no flat order
    ((2, 3, 70), "27x19", "sc", "fp16"),     # rows of one pair
    ((33, 7, 5), "27x19", "guo", "fp32"),    # a row one past a warp
    ((31, 9, 4), "27x19", "hcz", "bf16"),    # odd row, one node per thread in 16 bits
    ((65, 65, 3), "19x7", "sc", "fp32"),
    ((66, 11, 3), "27x19", "edm", "fp16"),   # pairs of nodes, 33 per row
    ((63, 1, 40), "15x7", "guo", "fp32"),    # planes of one row
    ((32, 32, 32), "27x19", "guo", "fp32"),  # less than one wave: the evenest blocks
    ((130, 34, 70), "27x27", "sc", "fp32"),
    ((225, 75, 9), "27x19", "edm", "fp16"),
])
def test_every_launch_gives_the_same_populations(shape, pair, forcing, storage):
    steps = 133   # two 64-step graphs and five eager steps: both AA parities last
    ref = _sim(shape, pair, forcing, storage)
    lbm.lbm_set_block(ref.h, 32, 1)
    ref.step(steps)
    f, g = ref.populations()
    runs = {"default": lambda s: None, "eager": lambda s: lbm.lbm_set_graphs(s.h, False),
            "tuned": lambda s: lbm.lbm_autotune(s.h, 1)}
    for name, setup in runs.items():
        sim = _sim(shape, pair, forcing, storage)
        setup(sim)
        sim.step(steps)
        f1, g1 = sim.populations()
        assert np.array_equal(f, f1) and np.array_equal(g, g1), name
        d = sim.diagnostics()
        fused = sim.step_diagnostics(1)
        for key in ("Ek", "Ep", "eps_k", "mass_f", "mass_g", "umax"):
            # both sum compensated FP32 terms of the same state (pair sums or raw deviations)
            assert fused[key] == pytest.approx(d[key], rel=1e-4 if key == "eps_k" else 1e-6), (name, key)
        sim.close()
    ref.close()

"""The diagnostics passes at the sizes where their launches change: planes of
one row, wraps in one and two planes, several planes per thread with a short
last run, and more step blocks than pass 2 adds up directly. Eqs. 22-26
against FP64 central differences and sums of the FP32 fields; the record fused
into a step, the standalone and the allocation-free one agree."""
import numpy as np
import pytest

import stgv_inputs as I
from paper_2605_14505_gb300 import lbm

from _helpers import lattice_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,pair,storage", [
    ((5, 1, 1), "19x7", "fp32"),
    ((7, 3, 2), "27x19", "fp32"),
    ((33, 9, 3), "27x19", "fp16"),
    ((130, 130, 101), "19x7", "fp32"),     # 5 planes per thread, 1 in the last run
    ((256, 64, 90), "27x19", "fp16"),      # pass-1 rows of more step blocks than are added up directly
])
@pytest.mark.parametrize("steps", [0, 1])
def test_records_match_the_fields(shape, pair, storage, steps):
    nx, ny, nz = shape
    p = lattice_params(nx, ny, nz, pair, "sc", 0.55, 0.6, 3e-3 / 1024, -3e-3 * 1024)
    sim = lbm.Simulation(p, storage=storage)
    sim.init_fields(*I.random_fields(nx, ny, nz, 6, 0.03, 0.01, 0.1))
    sim.step(steps)
    rho, u, rp = (a.reshape(-1, nz, ny, nx) for a in sim.fields())
    rho, rp = rho[0], rp[0]

    def d(f, axis):
        return 0.5 * (np.roll(f, -1, axis) - np.roll(f, 1, axis))

    cs2f, cs2g = (1 / 3, 0.25 if pair == "19x7" else 1 / 3)
    nu, D = cs2f * (p.tau_f - 0.5), cs2g * (p.tau_g - 0.5)
    gn2 = -p.G * p.rho0 / p.beta
    grad = sum(np.mean(d(rp, a) ** 2) for a in range(3))
    curl = (np.mean((d(u[2], 1) - d(u[1], 0)) ** 2) + np.mean((d(u[0], 0) - d(u[2], 2)) ** 2)
            + np.mean((d(u[1], 2) - d(u[0], 1)) ** 2))
    want = {"Ek": 0.5 * np.mean((u ** 2).sum(0)), "Ep": 0.5 * gn2 * np.mean(rp ** 2), "eps_p": D * gn2 * grad,
            "eps_k_curl": nu * curl, "mass_f": rho.sum(), "umax": np.sqrt((u ** 2).sum(0).max())}
    d0, d1 = sim.diagnostics(), lbm.lbm_diagnostics_noalloc(sim.h)
    d2, d3 = sim.diagnostics(), sim.step_diagnostics(1)
    assert d0 == d2                        # a fixed order of every sum
    for key, w in want.items():
        # FP32 terms (a dozen roundings of 6e-8 each) of compensated sums; rho in the fields rounds at 1
        assert d0[key] == pytest.approx(w, rel=2e-6), key
        assert d3[key] == pytest.approx(d0[key], rel=2e-6), key
        if key not in ("eps_p", "eps_k_curl"):
            assert d1[key] == pytest.approx(d0[key], rel=1e-9), key
    sim.close()

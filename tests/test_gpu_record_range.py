"""Record totals are FP64 beyond a thread's own sums: fields whose per-node
terms FP32 holds (up to 3.4e38) and whose sums it does not. eps_p overflows
FP32 within a block of the gradient pass in the first case; in the second E_p
does over the pass-1 rows and eps_p over the blocks. Both are finite in FP64.
A thread's FP32 terms take a dozen roundings of 6e-8 each."""
import numpy as np
import pytest

from paper_2605_14505_gb300 import lbm

from _helpers import lattice_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("amplitude,diffusivity", [(1e17, 1e3), (1e18, 0.1)])
def test_totals_beyond_fp32(amplitude, diffusivity):
    n = 32
    p = lattice_params(n, n, n, "19x7", "guo", 0.55, 0.5 + diffusivity / 0.25, 0.0, 0.0)
    sim = lbm.Simulation(p)
    rng = np.random.default_rng(9)
    rp = amplitude * (2 * rng.random(n ** 3) - 1)
    sim.init_fields(np.ones(n ** 3), np.zeros((3, n ** 3)), rp)
    got = sim.fields()[2].reshape(n, n, n)

    def d(axis):
        return 0.5 * (np.roll(got, -1, axis) - np.roll(got, 1, axis))

    ep = 0.5 * np.mean(got ** 2)
    eps_p = diffusivity * sum(np.mean(d(a) ** 2) for a in range(3))
    top = np.finfo(np.float32).max
    assert max(ep, eps_p) * n ** 3 > top > 10 * max(0.5 * np.max(got ** 2), diffusivity * 3 * amplitude ** 2)
    record = sim.diagnostics()
    assert record["Ep"] == pytest.approx(ep, rel=2e-6)
    assert record["eps_p"] == pytest.approx(eps_p, rel=2e-6)
    assert lbm.lbm_diagnostics_noalloc(sim.h)["Ep"] == pytest.approx(ep, rel=2e-6)
    fused = sim.step_diagnostics(1)
    assert fused["Ep"] == pytest.approx(ep, rel=2e-6)
    assert fused["eps_p"] == pytest.approx(eps_p, rel=2e-6)
    sim.close()

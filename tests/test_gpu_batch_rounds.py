"""The per-instance batch driver's rounds (instances that L2 holds together run
a call's steps before the next round's; one too large for it runs alone, in
skewed strips) and its records, taken on several streams: every instance's
fields and record equal, bit for bit, those of the same lattice on its own."""
import numpy as np
import pytest

from paper_2605_14505_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("calls", [(1,), (2, 3), (21, 70)])
def test_rounds_equal_single_lattices(calls):
    specs = [(88, "27x19", "sc"), (24, "19x7", "guo"), (84, "19x7", "sc"), (72, "27x19", "guo"), (33, "27x19", "edm"),
             (24, "27x19", "hcz"), (90, "27x19", "guo")]
    params = [lbm.lbm_params_from_physics(n, n, n, pair, fo, 100.0, 1.0, 1.0, 0.04) for n, pair, fo in specs]
    b = lbm.lbm_batch_create(params)
    lbm.lbm_batch_set_mode(b, "instances")
    lbm.lbm_batch_init_tgv(b, 3, 1e-3)
    for n in calls:
        lbm.lbm_batch_step(b, n)
    records = lbm.lbm_batch_diagnostics(b)
    for i, p in enumerate(params):
        n3 = p.nx ** 3
        rho, u, rp = lbm.lbm_get_fields(lbm.lbm_batch_instance(b, i), n3)
        sim = lbm.Simulation(p)
        sim.init_tgv(3, 1e-3)
        for _ in range(sum(calls)):
            sim.step(1)
        want = sim.fields()
        assert all(np.array_equal(x, y) for x, y in zip((rho, u, rp), want)), specs[i]
        assert records[i] == sim.diagnostics(), specs[i]
        sim.close()
    lbm.lbm_batch_destroy(b)

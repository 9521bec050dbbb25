"""Skewed strips on the GPU: lattices whose plans cut planes and rows, handles in
strips at the same time on streams of their own, the default streams. Bit for
bit the populations of whole-lattice steps (a call of one step runs whole).
tests/test_host_api.py checks that these plans are strips and their order."""
import numpy as np
import pytest

import stgv_inputs as I
from paper_2605_14505_gb300 import halo, lbm

from _helpers import lattice_params
from _strips import L2_BYTES, PLANS

pytestmark = pytest.mark.gpu


def _sim(shape, pair, storage, seed=8, forcing="sc"):
    sim = lbm.Simulation(lattice_params(*shape, pair, forcing, 0.55, 0.6, 3e-3 / 1024, -3e-3 * 1024), storage=storage)
    sim.init_fields(*I.random_fields(*shape, seed, 0.03, 0.01, 0.1))
    return sim


def _whole(shape, pair, storage, steps, seed=8, forcing="sc"):
    sim = _sim(shape, pair, storage, seed, forcing)
    for _ in range(steps):
        sim.step(1)
    sim.synchronize()
    return sim


def test_the_plans_are_those_of_this_device():
    import torch

    assert torch.cuda.get_device_properties(0).L2_cache_size == pytest.approx(L2_BYTES, rel=0.03)


@pytest.mark.parametrize("shape,pair,storage", [p[:3] for p in PLANS])
def test_strips_equal_whole_steps(shape, pair, storage):
    import torch

    calls = (19, 4, 37)
    whole = _whole(shape, pair, storage, sum(calls))
    strips = _sim(shape, pair, storage)
    for n in calls:
        strips.step(n)
    strips.synchronize()
    assert torch.equal(whole._store, strips._store)
    whole.close()
    strips.close()


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_strips_of_the_256_cubed_lattice(storage):
    """6 x 6 and 12 x 1 strips, a call that fills two groups and one that ends one early."""
    import torch

    p = lbm.lbm_params_from_physics(256, 256, 256, "27x19", "sc", 800.0, 0.1, 1.0, 0.04)
    whole, strips = (lbm.Simulation(p, storage=storage) for _ in range(2))
    for sim in (whole, strips):
        sim.init_tgv(1, 1e-3)
    for _ in range(37):
        whole.step(1)
    strips.step(32)
    strips.step(5)
    whole.synchronize()
    strips.synchronize()
    assert torch.equal(whole._store, strips._store)
    whole.close()
    strips.close()


def test_strips_of_planes_and_rows_from_a_graph():
    """128 eager steps, then replays from both parities."""
    import torch

    calls = (47, 90, 97, 33)
    whole = _whole((160, 160, 160), "19x7", "fp32", sum(calls), forcing="edm")
    strips = _sim((160, 160, 160), "19x7", "fp32", forcing="edm")
    for n in calls:
        strips.step(n)
    strips.synchronize()
    assert torch.equal(whole._store, strips._store)
    whole.close()
    strips.close()


def test_two_lattices_in_strips_at_once():
    import torch

    cases = [((160, 160, 160), "27x19", "fp32", 3), ((128, 96, 80), "27x19", "fp32", 4)]
    want = [_whole(*c[:3], 35, c[3]) for c in cases]
    got = [_sim(*c[:3], c[3]) for c in cases]
    for n in (20, 15):
        for sim in got:     # each on its own stream, neither waited for
            sim.step(n)
    for sim in got:
        sim.synchronize()
    for w, g in zip(want, got):
        assert torch.equal(w._store, g._store)
        w.close()
        g.close()


@pytest.mark.parametrize("stream", [0, 1, 2])   # null, legacy, per-thread
def test_strips_on_the_default_streams(stream):
    import torch

    for shape, pair, storage in (((128, 96, 80), "27x19", "fp32"), ((32, 32, 32), "19x7", "fp32")):
        whole = _whole(shape, pair, storage, 150)
        sim = _sim(shape, pair, storage)
        sim.synchronize()
        lbm.lbm_set_stream(sim.h, stream)
        sim.step(17)
        sim.step(133)
        record = sim.diagnostics()
        sim.synchronize()
        assert torch.equal(whole._store, sim._store)
        assert record == whole.diagnostics()
        whole.close()
        sim.close()


def test_one_rank_exchanges_with_itself():
    """SlabExchange with the library's backend, in a group of one rank: publish and
    follow order its copies around the odd steps."""
    nx, ny, nz = 48, 20, 12
    fields = [np.asarray(a).reshape(-1, nz, ny, nx) for a in I.random_fields(nx, ny, nz, 8, 0.03, 0.01, 0.1)[:3]]
    planes = np.arange(-1, nz + 1) % nz
    slab = lbm.Simulation(lattice_params(nx, ny, nz + 2, "27x19", "sc", 0.55, 0.6, 3e-3 / 1024, -3e-3 * 1024))
    rho, u, rp = (np.ascontiguousarray(f[:, planes]) for f in fields)
    slab.init_fields(rho.reshape(-1), u.reshape(3, -1), rp.reshape(-1))
    whole = _sim((nx, ny, nz), "27x19", "fp32")
    run = halo.SlabExchange(halo.LibrarySlab(slab), 0, 1)
    done = 0
    for n in (3, 4, 6):
        run.step(n)
        whole.step(n)
        done += n
        if done % 2:
            run.refresh_ghosts()
        for a, b in zip(slab.populations(), whole.populations()):
            a = np.asarray(a).reshape(-1, nz + 2, ny, nx)[:, 1:-1]
            assert np.array_equal(a, np.asarray(b).reshape(-1, nz, ny, nx)), done
    slab.close()
    whole.close()

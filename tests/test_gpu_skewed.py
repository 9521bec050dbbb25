"""Skewed stepping of lattices larger than L2 (strips of planes and rows run
several steps before the next strip) gives, bit for bit, the populations of
whole-lattice steps: cubes and flat or long boxes, strips along z alone and
along y and z, step counts that end a group early, start at either AA parity
and replay the two-group graph, every storage type. A CPU test walks the same
ranges over (y, z) and checks that no step runs before its neighbours'."""
import random

import pytest

import stgv_inputs as I
from paper_2605_14505_gb300 import lbm

from _helpers import lattice_params


def _range(n, strips, j, k, l, mirrored):
    """The library's skewed_range, restated."""
    first, count = 0, n
    if strips > 1:
        def cut(i):
            return i * n // strips + k - 1
        first = l if j == 0 else cut(j) - l
        count = (n + l if j == strips - 1 else cut(j + 1) - l) - first
        first -= n if first >= n else 0
    return (2 * n - first - count) % n if mirrored else first, count


def test_every_step_follows_its_neighbours():
    rng = random.Random(5)
    for _ in range(120):
        nz, ny, depth = rng.randint(1, 24), rng.randint(1, 24), rng.randint(1, 6)
        jz, jy = (max(1, min(rng.randint(1, 5), n // depth)) for n in (nz, ny))
        done = [[0] * ny for _ in range(nz)]
        steps = 0
        for group in range(3):
            k = rng.randint(1, depth)
            for z in range(jz):
                for y in range(jy):
                    for l in range(k):
                        z0, zn = _range(nz, jz, z, k, l, group % 2 == 1)
                        y0, yn = _range(ny, jy, y, k, l, group % 2 == 1)
                        assert 0 <= z0 < nz and 0 <= y0 < ny and 1 <= zn <= nz and 1 <= yn <= ny
                        cells = [((z0 + a) % nz, (y0 + b) % ny) for a in range(zn) for b in range(yn)]
                        for cz, cy in cells:
                            assert done[cz][cy] == steps + l
                            for dz in (-1, 0, 1):
                                for dy in (-1, 0, 1):
                                    # the neighbour's previous step is done, its next one is not
                                    assert done[(cz + dz) % nz][(cy + dy) % ny] in (steps + l, steps + l + 1)
                        for cz, cy in cells:
                            done[cz][cy] += 1
            steps += k
            assert all(v == steps for row in done for v in row)


@pytest.mark.gpu
@pytest.mark.parametrize("shape,pair,forcing,storage,calls", [
    ((82, 82, 82), "27x19", "sc", "fp32", (4, 5)),             # just too large for L2
    ((128, 96, 80), "27x19", "guo", "fp32", (1, 33, 16)),      # strips along z
    ((129, 97, 83), "19x7", "sc", "fp32", (17, 2, 4)),         # odd sides, flat launches
    ((256, 200, 34), "27x19", "edm", "fp32", (31, 20)),        # two strips of planes, the rest along y
    ((640, 150, 17), "19x7", "hcz", "fp32", (16, 15)),         # y alone
    ((40, 17, 530), "27x27", "sc", "fp32", (19,)),             # a long box
    ((4096, 300, 3), "27x19", "sc", "fp32", (18,)),            # too flat for z strips
    ((256, 256, 40), "27x19", "sc", "fp16", (21, 16)),         # pairs of nodes
    ((171, 160, 150), "19x7", "guo", "bf16", (18,)),           # one node per thread in 16 bits
    ((96, 96, 96), "27x19", "sc", "fp32", (47, 64, 97, 64)),   # into the graph, from both parities
])
def test_skewed_steps_equal_whole_lattice_steps(shape, pair, forcing, storage, calls):
    import torch

    nx, ny, nz = shape
    params = lattice_params(nx, ny, nz, pair, forcing, 0.55, 0.6, 3e-3 / 1024, -3e-3 * 1024)
    fields = I.random_fields(nx, ny, nz, 8, 0.03, 0.01, 0.1)
    whole, skewed = (lbm.Simulation(params, storage=storage) for _ in range(2))
    for sim in (whole, skewed):
        sim.init_fields(*fields)
    for n in calls:
        for _ in range(n):
            whole.step(1)          # a call of one step runs the whole lattice
        skewed.step(n)
    whole.synchronize()
    skewed.synchronize()
    assert torch.equal(whole._store, skewed._store)
    assert whole.step_count == skewed.step_count == sum(calls)
    whole.close()
    skewed.close()

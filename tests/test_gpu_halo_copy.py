"""lbm_halo_pack / lbm_halo_unpack byte for byte against the slot planes of the
raw store that the C header names, at sizes and buffer offsets of every copy
width (16, 4, 2 and 1 bytes), past one iteration of the kernel's four-wide
loop, and with both outgoing buffers the same memory."""
import pytest

from paper_2605_14505_gb300 import lbm

from _helpers import lattice_params

pytestmark = pytest.mark.gpu


def _runs(sim, sign):
    p = sim.params
    n3 = p.nx * p.ny * p.nz
    ef, eg = sim.velocity_sets()[0][0], sim.velocity_sets()[1][0]
    return [i * n3 for i, e in enumerate(ef) if e[2] == sign] + \
           [(sim.qf + i) * n3 for i, e in enumerate(eg) if e[2] == sign]


@pytest.mark.parametrize("shape,pair,storage,offset", [
    ((16, 12, 5), "27x19", "fp32", 0),      # 16-byte copies
    ((16, 12, 5), "27x19", "fp32", 4),      # the buffer allows 4
    ((33, 7, 4), "27x19", "fp16", 0),       # planes of 462 bytes: 2
    ((33, 7, 3), "19x7", "bf16", 1),        # an odd buffer address: 1
    ((201, 67, 3), "27x27", "fp32", 0),     # several strides of the four-wide loop and a remainder
])
def test_halo_copies_move_exactly_the_named_planes(shape, pair, storage, offset):
    import torch

    nx, ny, nz = shape
    sim = lbm.Simulation(lattice_params(nx, ny, nz, pair, "sc", 0.6, 0.6, 1e-5, -4.0), storage=storage)
    lbm.lbm_set_slab(sim.h, True)
    es = 4 if storage == "fp32" else 2
    plane = nx * ny * es
    g = torch.Generator(device="cuda").manual_seed(3)
    sim._store.random_(0, 256, generator=g)
    nbytes = lbm.lbm_halo_bytes(sim.h)
    lower, upper = (torch.zeros(nbytes + 32, dtype=torch.uint8, device="cuda") for _ in range(2))
    torch.cuda.synchronize()

    def expect(z, sign):
        return torch.cat([sim._store[r * es + z * plane:r * es + (z + 1) * plane] for r in _runs(sim, sign)])

    top = nz - 1
    for phase, (zl, sl), (zu, su) in ((0, (1, 1), (top - 1, -1)), (1, (0, -1), (top, 1))):
        lbm.lbm_halo_pack(sim.h, phase, lower.data_ptr() + offset, upper.data_ptr() + offset)
        sim.synchronize()
        for buf, z, sign in ((lower, zl, sl), (upper, zu, su)):
            assert torch.equal(buf[offset:offset + nbytes], expect(z, sign))
            assert not buf[offset + nbytes:].any() and not buf[:offset].any()
        # the same memory for both: the upper side's bytes stand
        lbm.lbm_halo_pack(sim.h, phase, upper.data_ptr() + offset, upper.data_ptr() + offset)
        sim.synchronize()
        assert torch.equal(upper[offset:offset + nbytes], expect(zu, su))
    for phase, (zl, sl), (zu, su) in ((0, (0, -1), (top, 1)), (1, (1, 1), (top - 1, -1))):
        before = sim._store.clone()
        lower.random_(0, 256, generator=g)
        upper.random_(0, 256, generator=g)
        torch.cuda.synchronize()
        lbm.lbm_halo_unpack(sim.h, phase, lower.data_ptr() + offset, upper.data_ptr() + offset)
        sim.synchronize()
        for buf, z, sign in ((lower, zl, sl), (upper, zu, su)):
            for k, r in enumerate(_runs(sim, sign)):
                at = r * es + z * plane
                before[at:at + plane] = buf[offset + k * plane:offset + (k + 1) * plane]
        assert torch.equal(sim._store, before)
    sim.close()

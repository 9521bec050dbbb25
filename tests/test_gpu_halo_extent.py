"""The extent check of the halo buffers against real allocations: a buffer that
ends with its allocation is taken, one that starts 16 bytes later is refused;
torch memory as before, at any offset that leaves room."""
import ctypes

import pytest

from paper_2605_14505_gb300 import lbm

from _helpers import lattice_params

pytestmark = pytest.mark.gpu


def _cudart():
    import torch

    torch.cuda.init()
    for name in ("libcudart.so.13", "/usr/local/cuda/lib64/libcudart.so"):
        try:
            return ctypes.CDLL(name)
        except OSError:
            pass
    pytest.fail("no CUDA runtime library")


def test_a_buffer_past_its_allocation_is_refused():
    import torch

    sim = lbm.Simulation(lattice_params(224, 224, 5, "27x19", "sc", 0.6, 0.6, 1e-5, -4.0))
    lbm.lbm_set_slab(sim.h, True)
    sim._store.zero_()
    torch.cuda.synchronize()
    nbytes = lbm.lbm_halo_bytes(sim.h)
    assert nbytes == 14 * 224 * 224 * 4
    rt, base, size = _cudart(), ctypes.c_void_p(), (3 << 20) + 512   # ends inside a 2 MiB page
    assert rt.cudaMalloc(ctypes.byref(base), ctypes.c_size_t(size)) == 0
    end = base.value + size - nbytes
    other = torch.zeros(nbytes + 4096, dtype=torch.uint8, device="cuda")
    for phase in (0, 1):
        for call in (lbm.lbm_halo_pack, lbm.lbm_halo_unpack):
            call(sim.h, phase, end, other.data_ptr())
            call(sim.h, phase, other.data_ptr() + 4096, end)
            for pair in ((end + 16, other.data_ptr()), (other.data_ptr(), end + 16)):
                with pytest.raises(lbm.LbmError) as ei:
                    call(sim.h, phase, *pair)
                assert ei.value.code == -1 and "shorter" in str(ei.value)
    sim.synchronize()
    sim.close()
    assert rt.cudaFree(base) == 0

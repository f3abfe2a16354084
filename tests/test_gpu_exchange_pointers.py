"""Device arrays that the exchange kernels cannot take themselves: at a byte
offset no float load reaches (the copy engine does the rows then), and pinned host
memory named by its device address.  The bytes are those of an aligned array."""
import ctypes

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16s", "bf16s"])
@pytest.mark.parametrize("vs,nx,ny", [("d2q9", 64, 32), ("d2q9", 33, 7), ("d2q7", 30, 90)])
@pytest.mark.parametrize("where", ["offset 1", "offset 2", "offset 4", "pinned"])
def test_arrays_the_kernels_cannot_reach(where, vs, nx, ny, storage):
    import torch
    from paper_1902_00530_gb300 import Lattice, Simulation
    q = 7 if vs == "d2q7" else 9
    sim = Simulation([Lattice(nx, ny, storage, 0, vs)], ["passive"], [dict(tau=1.0)])
    sim.init(1, [W.INIT_CONFIG2])
    sim.step(3)
    want = sim.get_state(host=True).numpy().copy()
    n = want.size * 4
    if where == "pinned":
        if storage == "f32":
            pytest.skip("an FP32 copy names its direction")
        buf, off = torch.zeros(n + 8, dtype=torch.uint8, pin_memory=True), 0
    else:
        buf, off = torch.zeros(n + 8, dtype=torch.uint8, device="cuda"), int(where.split()[1])
    torch.cuda.synchronize()
    ptr = ctypes.c_void_p(buf.data_ptr() + off)
    assert sim.lib.lbm_get_state(sim.ctx, 0, ptr, 0) == 0
    got = buf.cpu().numpy()
    np.testing.assert_array_equal(got[off:off + n].view(np.float32), want.ravel())
    assert not got[:off].any() and not got[off + n:].any()
    sim.step(3)
    assert (sim.get_state(host=True).numpy() != want).any()
    assert sim.lib.lbm_set_state(sim.ctx, 0, ptr, 0) == 0
    np.testing.assert_array_equal(sim.get_state(host=True).numpy(), want)
    sim.close()

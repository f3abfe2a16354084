"""State exchange and density steps at the widths and alignments where their
vector paths change: rows that hold whole 16-byte vectors, half of one, or none,
rows shorter than a warp, more rows than one pass of a block, a caller's
array at a 4-byte alignment, populations staged through the spare buffer in
several pieces.  Each result is compared with the definition, computed here."""
import numpy as np
import pytest

import workloads as W
from lbmtest import storage_shifts

pytestmark = pytest.mark.gpu
TORCH = {"f32": "float32", "f16s": "float16", "bf16s": "bfloat16"}


def _stored(f, storage, q):
    """What a lattice of this storage holds after being set to f, as FP32."""
    import torch
    t = torch.from_numpy(f)
    if storage == "f32":
        return f
    sh = torch.from_numpy(storage_shifts(storage, q)).float().view(q, 1, 1)
    return ((t - sh).to(getattr(torch, TORCH[storage])).float() + sh).numpy()


@pytest.mark.parametrize("storage", ["f32", "f16s", "bf16s"])
@pytest.mark.parametrize("q", [9, 7])
@pytest.mark.parametrize("nx,ny", [(1, 2), (30, 4), (36, 10), (64, 66), (1021, 6), (1032, 40), (4096, 14)])
def test_exchange_and_density_step(nx, ny, q, storage):
    import torch
    from paper_1902_00530_gb300 import Lattice, Simulation
    rng = np.random.default_rng(nx * 100 + ny)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4 if q == 9 else [0.5] + [1 / 12] * 6, np.float32)
    f = (w.reshape(-1, 1, 1) * rng.uniform(0.5, 1.5, (q, ny, nx))).astype(np.float32)
    want = _stored(f, storage, q)
    sim = Simulation([Lattice(nx, ny, storage, 0, "d2q9" if q == 9 else "d2q7")], ["passive"], [dict(tau=1.0)])
    sim.init(1, [W.INIT_CONFIG1])
    for host in (True, False):
        sim.init(1, [W.INIT_CONFIG1])
        sim.set_state(torch.from_numpy(f) if host else torch.from_numpy(f).cuda())
        np.testing.assert_array_equal(sim.get_state(host=True).numpy(), want)
        np.testing.assert_array_equal(sim.get_state().cpu().numpy(), want)
    odd = torch.empty(f.size + 1, dtype=torch.float32, device="cuda")[1:].view(q, ny, nx)  # 4-byte aligned
    sim.get_state(out=odd)
    np.testing.assert_array_equal(odd.cpu().numpy(), want)
    sim.set_state(odd)
    np.testing.assert_array_equal(sim.get_state(host=True).numpy(), want)
    # moments: the sums in FP32, so within a few roundings of their FP64 values
    rho, ux, uy = (t.cpu().numpy().astype(np.float64) for t in sim.moments())
    g = want.astype(np.float64)
    if q == 9:
        jx, jy = g[1] + g[5] + g[8] - g[3] - g[6] - g[7], g[2] + g[5] + g[6] - g[4] - g[7] - g[8]
    else:
        jx = g[1] - g[4] + 0.5 * (g[2] + g[6] - g[3] - g[5])
        jy = np.sqrt(0.75) * (g[2] + g[3] - g[5] - g[6])
    eps = 2.0 ** -24
    assert np.abs(rho - g.sum(0)).max() <= 8 * eps * g.sum(0).max()
    for u, j in ((ux, jx), (uy, jy)):
        assert np.abs(u - j / g.sum(0)).max() <= 16 * eps * (g.sum(0) / g.sum(0).min()).max()
    sim.add_density(0.01)
    c = np.float32(0.01 / q)
    np.testing.assert_array_equal(sim.get_state(host=True).numpy(), _stored(want + c, storage, q))
    sim.step(2)  # the spare buffer was only lent
    g = sim.get_state(host=True).numpy()
    assert np.isfinite(g).all() and abs(g.sum(dtype=np.float64) / (want + c).sum(dtype=np.float64) - 1) < 1e-2
    sim.close()

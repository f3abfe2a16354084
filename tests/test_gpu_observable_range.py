"""Observables over the range of densities that FP32 populations hold.  The sums are
formed in more than 24 bits, and at every scale: at 2^100 and more, where a sum in
FP32's range would overflow, around the bounds of the forms of rho^2 and of the sums of
rho, with zero and tiny densities in the same rows, from one lattice to the next.

The state is at rest (populations w_i rho, symmetric, so that j is exactly zero): the
records are the sums of rho alone, compared with the same sums of the stored
populations in exact integer arithmetic."""
from fractions import Fraction

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
# one FP32 rounding per addition of a site's populations, and what the sums add
TOL = 16 * 2.0 ** -24


def _exact(f):
    """(mass, drho_y, drho_x, var_rho) of FP32 populations, sums exact."""
    rho = np.vectorize(lambda *v: sum(map(Fraction, map(float, v))), otypes=[object])(*f)
    ny, nx = rho.shape
    mass, mean = rho.sum(), rho.sum() / (nx * ny)
    std = lambda m: float(sum((x - mean) ** 2 for x in m) / len(m)) ** 0.5  # noqa: E731
    return float(mass), std(rho.sum(0) / ny), std(rho.sum(1) / nx), float(sum((rho - mean).ravel() ** 2) / (nx * ny))


@pytest.mark.parametrize("vs,vec,nx,ny", [("d2q9", 4, 160, 24), ("d2q9", 1, 33, 40), ("d2q7", 2, 70, 36)])
@pytest.mark.parametrize("lo,hi", [(0, 0), (-60, -45), (-52, -48), (45, 62), (56, 61), (94, 98), (108, 118), (118, 124),
                                   (-120, 120), (-140, -100)])
def test_records_at_every_scale(lo, hi, vs, vec, nx, ny):
    _check(lo, hi, vs, vec, 8, nx, ny)


@pytest.mark.parametrize("lo,hi", [(49, 50), (59, 59), (95, 96)])
def test_records_of_tall_strips(lo, hi):
    """One lane adds a thousand rows: the squares just below a bound must not add up past FP32."""
    _check(lo, hi, "d2q9", 1, 1024, 32, 1024)


def _check(lo, hi, vs, vec, rows, nx, ny):
    import torch
    from paper_1902_00530_gb300 import Lattice, Simulation
    q = 7 if vs == "d2q7" else 9
    rng = np.random.default_rng(100 * abs(lo) + abs(hi) + nx)
    scale = np.exp2(rng.integers(lo, hi + 1, (ny, nx)).astype(np.float64))
    rho = rng.uniform(1.0, 2.0, (ny, nx)) * scale
    if (lo, hi) == (-120, 120):
        rho[rng.random((ny, nx)) < 0.2] = 0.0
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4 if q == 9 else [0.5] + [1 / 12] * 6)
    f = (w.reshape(-1, 1, 1) * rho).astype(np.float32)
    assert np.isfinite(f).all()
    sim = Simulation([Lattice(nx, ny, "f32", 0, vs)], ["passive"], [dict(tau=1.0)])
    sim.set_tuning(1, vec, rows, 4, 0)
    sim.init(1, [W.INIT_CONFIG1])
    sim.set_state(torch.from_numpy(f))
    got = sim.observables()
    sim.close()
    mass, sy, sx, var = _exact(f)
    top = float(rho.max())
    assert abs(got["mass"] - mass) <= TOL * mass
    assert got["phi"] == 0.0 and got["zeta"] == 0.0
    assert abs(got["drho_y"] - sy) <= TOL * top and abs(got["drho_x"] - sx) <= TOL * top
    assert abs(got["var_rho"] - var) <= TOL * top * top


@pytest.mark.parametrize("tuning", [(4, 8, 4, 0), (1, 8, 4, 0), (4, 8, 4, 3)], ids=str)
@pytest.mark.parametrize("vs", ["d2q9", "d2q7"])
@pytest.mark.parametrize("power", [0, 55, 96, 118])
def test_sampled_steps_of_a_uniform_state(power, vs, tuning):
    """A uniform state at rest stays itself, whatever its scale: the records that
    the step kernels' own sums give, over strips that end inside the lattice."""
    import torch
    from paper_1902_00530_gb300 import Lattice, Simulation
    q, nx, ny = (7 if vs == "d2q7" else 9), 160, 28
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4 if q == 9 else [0.5] + [1 / 12] * 6)
    f = np.broadcast_to((w * 1.25 * 2.0 ** power).astype(np.float32).reshape(q, 1, 1), (q, ny, nx)).copy()
    sim = Simulation([Lattice(nx, ny, "f32", 0, vs)], ["passive"], [dict(tau=1.0)], sample_every=2, ring_capacity=4)
    sim.set_tuning(1, *tuning)
    sim.init(1, [W.INIT_CONFIG1])
    sim.set_state(torch.from_numpy(f))
    sim.step(4)
    mass = 1.25 * 2.0 ** power * nx * ny
    records = sim.observable_series(0)
    assert [r["t"] for r in records] == [2, 4]
    for r in records:
        assert abs(r["mass"] - mass) <= 4 * TOL * mass
        assert r["phi"] <= TOL and r["zeta"] >= -TOL and r["var_rho"] <= TOL * (1.25 * 2.0 ** power) ** 2
    sim.close()

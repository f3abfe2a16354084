"""The resident launch (small lattices held in the shared memory of a cluster
for a whole stretch of steps) against one launch per step.

Both run the same per-site operations, so every state must be bitwise the
same: at the edges of the row bands (heights that no cluster size divides, the
two-row bands MIPS needs at least, a lattice of one block), of the halo (widths
1, 2 and odd ones, a band wider than a block's threads), over the closures,
storage types, noise on and off in one group, both lattices, odd and even
stretches (the last step then writes the other buffer, or the one the first
read), and between sample steps.
"""
import numpy as np
import pytest

import workloads as W
from lbmtest import split_preset

pytestmark = pytest.mark.gpu
SEED = W.seed(12)


def _run(persistent, storage, cfg, calls, every=0, graphs=True):
    from paper_1902_00530_gb300 import Lattice, Simulation
    lats, mods, prms, specs = [], [], [], []
    for k, (nx, ny, name, over, init, vs) in enumerate(cfg):
        model, d = split_preset(name, **over)
        lats.append(Lattice(nx, ny, storage, k, vs))
        mods.append(model)
        prms.append(d)
        specs.append(init)
    sim = Simulation(lats, mods, prms, sample_every=every, ring_capacity=64 if every else 0)
    sim.set_persistent(persistent)
    sim.set_graphs(graphs)
    sim.init(SEED, specs)
    launches = []
    for n in calls:
        sim.step(n)
        launches.append(sim.last_launch_count())
    out = [sim.get_state(k, host=True).numpy() for k in range(len(cfg))]
    series = [sim.observable_series(k) for k in range(len(cfg))] if every else None
    sim.close()
    return out, launches, series


def _fits(q, storage, preset, nx, ny):
    """Whether some cluster of up to 16 blocks holds the lattice: two buffers of
    the tallest band with its halo, and the MIPS densities, in 227 KB each."""
    mips = preset.startswith("MIPS")
    halo, eb = (2 if mips else 1), (4 if storage == "f32" else 2)
    for c in range(1, 17):
        rows, np_ = -(-ny // c), nx + 2
        size = 2 * q * (rows + 2 * halo) * np_ * eb + (16 + (rows + 2) * np_ * 4 if mips else 0)
        if ny // c >= halo and size <= 232448:
            return True
    return False


def _same(storage, cfg, calls=(7, 6), every=0, graphs=True, fits=True):
    a, la, sa = _run("auto", storage, cfg, calls, every, graphs)
    b, lb, sb = _run(0, storage, cfg, calls, every, graphs)
    for k, (x, y) in enumerate(zip(a, b)):
        np.testing.assert_array_equal(x, y, err_msg=f"lattice {k}")
    if fits and max(n[0] * n[1] for n in cfg) <= SURE:
        assert all(p < q for p, q in zip(la, lb)), (la, lb)  # the stretches ran as one launch each
    if every:
        for x, y in zip(sa, sb):
            assert [r["t"] for r in x] == [r["t"] for r in y]
    return la


C2 = W.INIT_CONFIG2
# sites up to which a lattice that fits runs resident for certain (several times faster than the
# other forms); beyond, the tuner's timings decide.  [2, 2]: the stretch and the time advance,
# [8, 7]: its steps and the time advance.
SURE = 10800
SIZES9 = [(64, 64), (1, 7), (2, 5), (33, 2), (90, 31), (801, 20), (200, 150)]
SIZES7 = [(90, 30), (1, 8), (2, 6), (33, 4), (180, 60), (801, 22), (180, 150)]


@pytest.mark.parametrize("storage", ["f32", "f16s", "bf16s"])
@pytest.mark.parametrize("preset", ["MIPS_RHO1", "CIL_RHO1", "PASSIVE"])
@pytest.mark.parametrize("size", SIZES9, ids=lambda s: f"{s[0]}x{s[1]}")
def test_resident_equals_per_step_d2q9(size, preset, storage):
    fits = _fits(9, storage, preset, *size)
    launches = _same(storage, [(*size, preset, {}, C2, "d2q9")], fits=fits)
    assert launches in ([[2, 2]] if fits and size[0] * size[1] <= SURE else [[2, 2], [8, 7]] if fits else [[8, 7]])


@pytest.mark.parametrize("storage", ["f32", "bf16s"])
@pytest.mark.parametrize("preset", ["MIPS_Q7_RHO1", "CIL_Q7_RHO1", "PASSIVE"])
@pytest.mark.parametrize("size", SIZES7, ids=lambda s: f"{s[0]}x{s[1]}")
def test_resident_equals_per_step_d2q7(size, preset, storage):
    fits = _fits(7, storage, preset, *size)
    launches = _same(storage, [(*size, preset, {}, C2, "d2q7")], fits=fits)
    assert launches in ([[2, 2]] if fits and size[0] * size[1] <= SURE else [[2, 2], [8, 7]] if fits else [[8, 7]])


@pytest.mark.parametrize("graphs", [True, False])
@pytest.mark.parametrize("every", [0, 5])
def test_resident_batch_of_groups(every, graphs):
    """Groups of both lattices and closures in one batch, lattices of different
    sizes in a group, noise in some of them only, more lattices than fit the
    GPU at once, sample steps between the stretches."""
    cfg = [(64, 48, "CIL_RHO1", dict(sigma=0.0 if k % 3 else 0.05), C2, "d2q9") for k in range(40)]
    cfg += [(97, 33, "CIL_RHO1", {}, C2, "d2q9"), (64, 64, "MIPS_RHO1", {}, W.INIT_CONFIG1, "d2q9"),
            (180, 60, "CIL_Q7_RHO1", {}, C2, "d2q7"), (90, 30, "MIPS_Q7_RHO1", {}, W.INIT_CONFIG1, "d2q7")]
    _same("f32", cfg, calls=(13, 12), every=every, graphs=graphs)


def test_lattice_beyond_a_cluster_stays_per_step():
    """A lattice whose two buffers exceed the shared memory of sixteen blocks."""
    la = _run("auto", "f32", [(400, 400, "CIL_RHO1", {}, C2, "d2q9")], (6,))[1]
    assert la == [7]  # six steps and the time advance


@pytest.mark.parametrize("storage", ["f32", "f16s"])
@pytest.mark.parametrize("preset,vs", [("MIPS_RHO1", "d2q9"), ("CIL_RHO1", "d2q9"), ("PASSIVE", "d2q9"),
                                       ("MIPS_Q7_RHO1", "d2q7"), ("CIL_Q7_RHO1", "d2q7")])
@pytest.mark.parametrize("size", [(1021, 402), (1022, 300), (1923, 130), (257, 640), (4099, 514)],
                         ids=lambda s: f"{s[0]}x{s[1]}")
def test_tuned_plain_shapes_equal_one_site_per_thread(size, preset, vs, storage):
    """Widths that no vector divides, beyond the resident launch: the tuned
    shape of plain steps (short strips, vectors that a row ends inside)
    against one site per thread in 8-row strips."""
    from paper_1902_00530_gb300 import Lattice, Simulation
    model, d = split_preset(preset)
    out = []
    for fixed in (False, True):
        sim = Simulation([Lattice(*size, storage, 3, vs)], [model], [d])
        if fixed:
            sim.set_tuning(1, 1, 8, 4, 0)
        sim.init(SEED, [C2])
        sim.step(5)
        out.append(sim.get_state(host=True).numpy())
        sim.close()
    np.testing.assert_array_equal(out[0], out[1])

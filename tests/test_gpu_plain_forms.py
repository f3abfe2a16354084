"""Every form that steps without a sample can run in, pinned, against one launch per
step of one site per thread in 8-row strips: states must be bitwise the same.

Direct shapes: every vector of a storage type at widths below it and at each
remainder, strips of 1, 2, 4 and 8 rows with a shorter last one, with noise and
without.  Resident launches: every cluster size that holds the lattice.  The forms
are read back, and the resident launches counted, so no case can pass in
another form."""
import numpy as np
import pytest

import workloads as W
from lbmtest import split_preset

pytestmark = pytest.mark.gpu
SEED = W.seed(21)
MODELS = [("MIPS_RHO1", "d2q9"), ("CIL_RHO1", "d2q9"), ("PASSIVE", "d2q9"),
          ("MIPS_Q7_RHO1", "d2q7"), ("CIL_Q7_RHO1", "d2q7"), ("PASSIVE", "d2q7")]


def _sim(lattices, every=0):
    """lattices: (nx, ny, storage, preset, overrides, velocity set) each."""
    from paper_1902_00530_gb300 import Lattice, Simulation
    lats, mods, prms = [], [], []
    for k, (nx, ny, storage, preset, over, vs) in enumerate(lattices):
        model, d = split_preset(preset, **over)
        lats.append(Lattice(nx, ny, storage, k, vs))
        mods.append(model)
        prms.append(d)
    sim = Simulation(lats, mods, prms, sample_every=every, ring_capacity=16 if every else 0)
    sim.set_tuning(1, 1, 8, 4, 0)
    return sim


def _run(sim, form, n):
    """States, launch count and form after n steps from the initial state."""
    sim.set_plain_form(*form)
    sim.init(SEED, [W.INIT_CONFIG2] * len(sim.lattices))
    sim.step(n)
    return ([sim.get_state(k, host=True).numpy().copy() for k in range(len(sim.lattices))], sim.last_launch_count(),
            sim.get_plain_form())


@pytest.mark.parametrize("storage,vec", [(s, v) for s in ("f32", "f16s", "bf16s") for v in (1, 2, 4, 8)
                                         if not (s == "f32" and v == 8)])
@pytest.mark.parametrize("preset,vs", MODELS, ids=lambda v: str(v))
def test_direct_shapes(preset, vs, storage, vec):
    # widths below the vector, one strip and a bit, two strips and each remainder
    widths = sorted({1, max(1, vec - 1), vec, vec + 1} | {32 * vec + r for r in range(vec + 1)} | {64 * vec + vec // 2 + 1})
    for sigma in (0.05, 0.0):
        if preset == "PASSIVE" and sigma == 0.0 and vec == 1:
            continue
        for nx in widths:
            sim = _sim([(nx, 10, storage, preset, dict(sigma=sigma), vs)])
            ref = _run(sim, (0,), 3)[0][0]
            for rows in (1, 2, 4, 8):
                if vs == "d2q7" and rows == 1:
                    continue
                got, launches, form = _run(sim, (1, vec, rows, 4), 3)
                assert form == (1, vec, rows, 4) and launches == 4  # three steps and the time advance
                np.testing.assert_array_equal(got[0], ref, err_msg=f"nx {nx} rows {rows} sigma {sigma}")
            sim.close()


@pytest.mark.parametrize("every", [0, 3])
@pytest.mark.parametrize("storage", ["f32", "bf16s"])
@pytest.mark.parametrize("vs", ["d2q9", "d2q7"])
def test_group_of_whole_and_ragged_widths(vs, storage, every):
    """Rows that end inside a vector beside rows that do not, noise in some lattices
    only, more rows than blocks hold, and steps that take a sample in between."""
    q7 = "_Q7" if vs == "d2q7" else ""
    lats = [(256, 48, storage, f"CIL{q7}_RHO1", {}, vs), (131, 20, storage, f"CIL{q7}_RHO1", dict(sigma=0.0), vs),
            (67, 64, storage, f"CIL{q7}_RHO1", {}, vs), (130, 34, storage, f"MIPS{q7}_RHO1", {}, vs)]
    sim = _sim(lats, every)
    ref = _run(sim, (0,), 11)[0]
    series = [sim.observable_series(k) for k in range(4)] if every else None
    for form in ((1, 2, 2, 8), (1, 4, 4, 4), (1, 4, 16, 8)):
        got = _run(sim, form, 11)[0]
        for k in range(4):
            np.testing.assert_array_equal(got[k], ref[k], err_msg=f"lattice {k} form {form}")
            if every:
                assert sim.observable_series(k) == series[k]
    sim.close()


@pytest.mark.parametrize("storage", ["f32", "f16s", "bf16s"])
@pytest.mark.parametrize("preset,vs", MODELS, ids=lambda v: str(v))
@pytest.mark.parametrize("size", [(1, 6), (3, 34), (90, 30), (64, 50), (801, 22), (200, 150)],
                         ids=lambda s: f"{s[0]}x{s[1]}")
def test_resident_clusters(size, preset, vs, storage):
    from paper_1902_00530_gb300 import LBMError
    nx, ny = size
    q, eb, halo = (7 if vs == "d2q7" else 9), (4 if storage == "f32" else 2), (2 if preset.startswith("MIPS") else 1)
    for sigma in (0.05, 0.0):
        sim = _sim([(nx, ny, storage, preset, dict(sigma=sigma), vs)])
        ref = {n: _run(sim, (0,), n)[0][0] for n in (4, 5)}
        ran = 0
        for c in range(1, 17):
            rows = -(-ny // c)
            size_b = -(-2 * q * (rows + 2 * halo) * (nx + 2) * eb // 16) * 16 + ((rows + 2) * (nx + 2) * 4 if halo == 2 else 0)
            if ny // c < halo or size_b > 232448:
                with pytest.raises(LBMError):
                    sim.set_plain_form(2, c)
                continue
            for n in (4, 5):
                got, launches, form = _run(sim, (2, c), n)
                assert form == (2, c, 0, 0) and launches == 2
                np.testing.assert_array_equal(got[0], ref[n], err_msg=f"cluster {c}, {n} steps, sigma {sigma}")
            ran += 1
        # (wide MIPS bands of two rows with their four halo rows exceed a block in FP32)
        assert ran > 0 or (nx, halo, eb) == (801, 2, 4), "no cluster ran"
        sim.close()


def test_refused_forms():
    from paper_1902_00530_gb300 import LBMError
    sim = _sim([(64, 48, "f32", "CIL_RHO1", {}, "d2q9"), (60, 30, "f32", "CIL_Q7_RHO1", {}, "d2q7")])
    for form in ((3, 1, 8, 4), (-1,), (1, 8, 8, 4), (1, 3, 8, 4), (1, 4, 0, 4), (1, 4, 3, 4), (1, 4, 8, 9), (2, 0), (2, 17)):
        with pytest.raises(LBMError):
            sim.set_plain_form(*form)
        assert sim.get_plain_form() == (0, 0, 0, 0)
    sim.set_plain_form(1, 4, 2, 4)
    sim.set_tuning(1, 1, 8, 4, 0)
    assert sim.get_plain_form(1) == (0, 0, 0, 0)
    sim.set_tuning(0)
    with pytest.raises(LBMError):
        sim.set_plain_form(1, 4, 2, 4)  # the shape of sample steps is not fixed
    sim.close()

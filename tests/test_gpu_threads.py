"""Two host threads, each with a context of its own, stepping lattices of
different size with the same kernel.  The largest dynamic shared memory a kernel
may be launched with is a property of the kernel, common to all threads: a
launcher that lowered it for its own lattice would make the other thread's next
launch fail.  Every call must succeed and every state be that of a run alone."""
import threading

import numpy as np
import pytest

import workloads as W
from lbmtest import split_preset

pytestmark = pytest.mark.gpu

CALLS = 1500


def _sim(size, preset, vs, storage, tuning):
    from paper_1902_00530_gb300 import Lattice, Simulation
    model, d = split_preset(preset)
    sim = Simulation([Lattice(*size, storage, 0, vs)], [model], [d])
    if tuning:
        sim.set_tuning(1, *tuning)
    sim.set_graphs(False)  # every call launches the kernel itself
    sim.init(W.seed(3), [W.INIT_CONFIG2])
    sim.step(2)  # automatic tuning, where it is on, happens here
    return sim


@pytest.mark.parametrize("preset,vs,storage,small,large", [
    # lattices that run resident for certain: 20 and 61 KB of shared memory a block
    ("CIL_Q7_RHO1", "d2q7", "f32", ((90, 30), None), ((180, 60), None)),
    # staged rings of 3 and 8 rows
    ("CIL_RHO1", "d2q9", "f32", ((256, 64), (4, 16, 4, 3)), ((256, 64), (4, 16, 4, 8))),
    ("CIL_Q7_RHO1", "d2q7", "bf16s", ((256, 64), (8, 16, 4, 3)), ((256, 64), (8, 16, 4, 8))),
], ids=["resident", "staged", "staged_q7"])
def test_contexts_of_two_threads_are_independent(preset, vs, storage, small, large):
    errors, states = [], {}

    def work(key, sim):
        try:
            for _ in range(CALLS):
                sim.step(2)
            states[key] = sim.get_state(host=True).numpy()
        except Exception as e:  # noqa: BLE001 -- reported by the assertion below
            errors.append((key, repr(e)))

    sims = {key: _sim(size, preset, vs, storage, tuning) for key, (size, tuning) in (("s", small), ("l", large))}
    ts = [threading.Thread(target=work, args=kv) for kv in sims.items()]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for sim in sims.values():
        sim.close()
    assert not errors, errors
    for key, (size, tuning) in (("s", small), ("l", large)):
        sim = _sim(size, preset, vs, storage, tuning)
        sim.step(2 * CALLS)
        np.testing.assert_array_equal(states[key], sim.get_state(host=True).numpy(), err_msg=key)
        sim.close()

"""What choosing the plain form costs: a width that no vector divides has ten shapes
for its sample steps (one site per thread), and its tuning must not be dominated by
the shapes that only steps without a sample may have.  A timing lasts a quarter of a
millisecond, or half of that for a plain shape, and up to as much again to warm up and to
find its length, so the bound is on the number of timings."""
import time

import pytest

import workloads as W
from lbmtest import gpu_sim, split_preset

pytestmark = pytest.mark.gpu
TIMINGS = 10 + 10 + 8  # own shapes, plain shapes, the final look


@pytest.mark.parametrize("preset,storage", [("PASSIVE", "bf16s"), ("CIL_RHO1", "f32")])
def test_tuning_an_odd_width(preset, storage):
    model, d = split_preset(preset)
    sim = gpu_sim(model, d, 1021, 777, W.seed(1), W.INIT_CONFIG2, storage=storage)
    sim.tune()  # loads the kernels
    best = 1e9
    for _ in range(7):
        t = time.perf_counter()
        sim.tune()
        best = min(best, time.perf_counter() - t)
    sim.close()
    print(f"{preset} {storage}: {best * 1e3:.1f} ms")
    assert best < TIMINGS * 0.5e-3

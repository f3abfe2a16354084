"""Destroying a context while another stream is being captured in the global mode,
which refuses memory calls to every thread: a refused one also ends the capture
in an error, and a context may own pinned memory by then.  (Calls that wait for
their stream are refused in that time whatever they do.)"""
import pytest

import workloads as W
from lbmtest import gpu_sim, split_preset

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("observed", [False, True])
def test_destroy_while_another_stream_is_captured(observed):
    import torch
    model, d = split_preset("CIL_RHO1")
    sim = gpu_sim(model, d, 64, 48, W.seed(1), W.INIT_CONFIG2)
    if observed:
        assert sim.observables()["t"] == 0
    sim.synchronize()
    x = torch.zeros(16, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="global"):
        x += 1
        sim.close()
        x += 1
    g.replay()
    torch.cuda.synchronize()
    assert (x.cpu().numpy() == 2).all()

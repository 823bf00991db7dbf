"""An error that one call returned is not reported again by the next: the
read-backs (lb_heat_flux, lb_sync, lb_get_state and lb_set_state on the device,
the batch's) return the status of their own launch, not the runtime's record
of the last failure. The failure here is a call on a stream under capture, which
synchronises and is refused by the runtime without anything having run."""

import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

RELAXED = 2  # cudaStreamCaptureModeRelaxed


def refused_under_capture(stream, call):
    rt = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
    graph = ctypes.c_void_p()
    s = ctypes.c_void_p(stream.cuda_stream)
    assert rt.cudaStreamBeginCapture(s, RELAXED) == 0
    try:
        with pytest.raises(Exception):
            call()
    finally:
        rt.cudaStreamEndCapture(s, ctypes.byref(graph))  # invalidated by the refusal
        rt.cudaGetLastError()
    assert not graph.value


def test_read_backs_after_a_refused_call():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1501_03857_gb300 import lb
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        sim = lb.Simulation(lb.Config(Lx=40, Ly=24, pool_height=10.0), superheat=0.01, stream=stream)
        batch = lb.Batch([{"cfg": lb.Config(Lx=40, Ly=24, pool_height=10.0), "superheat": 0.01}], stream=stream)
        f, th = torch.empty(9, 24, 40, device="cuda"), torch.empty(24, 40, device="cuda")
        calls = {"heat_flux": sim.heat_flux, "sync": sim.sync, "batch": batch.heat_flux,
                 "get": lambda: lb.check(lb.lib.lb_get_state(sim.h, f.data_ptr(), th.data_ptr(), 1)),
                 "set": lambda: lb.check(lb.lib.lb_set_state(sim.h, f.data_ptr(), th.data_ptr(), 1))}
        sim.step(3)
        batch.step(3)
        want = sim.heat_flux()
        for name, call in calls.items():
            refused_under_capture(stream, sim.heat_flux)
            got = call()  # raised the refusal's error again
            if name == "heat_flux":
                assert got == want
            if name == "batch":
                assert got["q_inst"][0] == want["q_inst"]
        assert np.array_equal(f.cpu().numpy(), sim.get_state()[0])
        sim.close()
        batch.close()

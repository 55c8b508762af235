"""A step launch that the runtime refuses is reported by that call alone. The refusal
here is the host's: a launch on the legacy default stream while another stream
is being captured in global mode."""
import ctypes as C

import numpy as np
import pytest

from paper_2401_17183_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    from paper_2401_17183_gb300 import build as B
    B.build()
    from paper_2401_17183_gb300 import vlb
    vlb.load()
    return vlb


@pytest.mark.parametrize("kind,steps", [("single steps", 1), ("cluster", 2), ("cooperative", 2), ("d3q39", 1)])
def test_refused_launch_is_not_reported_twice(V, kind, steps):
    mesh = {"single steps": lambda: W.channel_mesh(8, 8, 40, stretch=0.5, bump=0.02),
            "cluster": lambda: W.channel2d_mesh(16, 64, stretch=0.5),
            "cooperative": lambda: W.channel2d_mesh(80, 80, stretch=0.5),
            "d3q39": lambda: W.periodic_sine_mesh3d(8, 0.01, q=39)}[kind]()
    rho, u = W.noise_fields(mesh, amp=0.01, seed=4)
    s = V.Sim(V.Mesh(mesh), W.params(0.8), rho, u, precision=V.VLB_F64 if kind == "d3q39" else V.VLB_F32)
    s.step(steps)
    s.sync()
    cu = C.CDLL("libcuda.so.1")
    stream, graph = C.c_void_p(), C.c_void_p()
    assert cu.cuStreamCreate(C.byref(stream), 0) == 0          # a stream that the legacy one waits for
    assert cu.cuStreamBeginCapture_v2(stream, 0) == 0          # CU_STREAM_CAPTURE_MODE_GLOBAL
    with pytest.raises(V.VlbError) as e:
        s.step(steps)
    assert e.value.code == "ECUDA"
    cu.cuStreamEndCapture(stream, C.byref(graph))              # (the refusal has ended it)
    cu.cuStreamDestroy_v2(stream)
    s.reset(rho, u)                                            # a valid call again
    s.step(steps)
    a = s.get_state()
    t = V.Sim(s.mesh, W.params(0.8), rho, u, precision=V.VLB_F64 if kind == "d3q39" else V.VLB_F32)
    t.step(steps)
    assert np.array_equal(a, t.get_state())

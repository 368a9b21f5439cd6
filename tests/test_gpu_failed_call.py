"""A call that a CUDA error ends says so once and leaves the next calls, of its handle and of
others, alone.  The error is made on the host: the handle's stream is being captured, where a
synchronising read is refused."""
import ctypes

import numpy as np
import pytest

from paper_2511_15908_gb300 import scenes

from test_gpu_parity import sph  # noqa: F401

pytestmark = pytest.mark.gpu


def read_under_capture(sph, sim, x, v):  # noqa: F811
    """A state read into x and v that fails; the capture is over afterwards."""
    f32p = ctypes.POINTER(ctypes.c_float)
    cuda, stream, graph = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(sim.stream.cuda_stream), ctypes.c_void_p()
    assert cuda.cuStreamBeginCapture_v2(stream, 1) == 0                     # thread-local
    st = sim.L.sph_get_state(sim.h, x.ctypes.data_as(f32p), v.ctypes.data_as(f32p), None, None, None)
    ended = cuda.cuStreamEndCapture(stream, ctypes.byref(graph))
    assert st == sph.ERR_CUDA and ended != 0


@pytest.mark.parametrize("then", ["read", "step", "other"])
def test_next_call_after_a_failed_one(sph, then):  # noqa: F811
    sc = scenes.tiny(seed=1, n=(4, 4, 4))
    sim, ref = sph.Simulation(sc), sph.Simulation(sc)
    sim.step(1)
    ref.step(1)
    sim.sync()
    x, v = np.empty((sim.n, 3), np.float32), np.empty((sim.n, 3), np.float32)
    read_under_capture(sph, sim, x, v)
    if then == "step":
        sim.step(1)
        ref.step(1)
    elif then == "other":
        other = sph.Simulation(sc)
        other.step(1)
        other.close()
    np.testing.assert_array_equal(sim.state()["x"], ref.state()["x"])
    sim.close()
    ref.close()

"""Grids small enough for whole steps in one cluster launch run their collide-stream pass as
its own kernel when a form of it was asked for (lbm_set_collide_form), so that
lbm_path_flags names what runs.  Counted in a captured lone step: one launch, or four."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def launches_of_a_step(sim, stream):
    """Graph nodes of one lone step, by capturing it (it does not run)."""
    drv = C.CDLL("libcuda.so.1")
    graph, n, h = C.c_void_p(), C.c_size_t(), C.c_void_p(stream.cuda_stream)
    assert drv.cuStreamBeginCapture_v2(h, 1) == 0  # thread-local
    sim.step_async(1)
    assert drv.cuStreamEndCapture(h, C.byref(graph)) == 0
    assert drv.cuGraphGetNodes(graph, None, C.byref(n)) == 0
    assert drv.cuGraphDestroy(graph) == 0
    return n.value


def test_asked_form_runs(cuda):
    from paper_1906_09530_gb300 import Simulation, lbm_maxwell
    from paper_1906_09530_gb300 import workloads as W
    rg, rl = lbm_maxwell(0.6)
    rho = W.drop(128, 64, rg, rl, 16.0, 8.0)
    s = cuda.cuda.Stream()
    out = []
    for form, launches, flags in ((0, 1, 0), (8, 4, 4), (-1, 4, 0), (0, 1, 0)):
        sim = Simulation(128, 64, 0.6, 0.1, 1.0, 0.5, precision="mixed", stream=s)
        sim.set_launch_mode(0, 0, 0)  # lone steps by direct launches
        sim.set_collide_form(8)
        sim.set_collide_form(form)
        assert sim.path_flags == flags
        sim.set_fields(rho)
        sim.step(5)
        out.append(sim.get_populations()[0])
        cuda.cuda.synchronize()
        assert launches_of_a_step(sim, s) == launches
        sim.close()
    assert all(np.array_equal(f, out[0]) for f in out[1:])

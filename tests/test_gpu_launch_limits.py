"""The dynamic shared memory that a kernel may use is state of the device, shared by all
grids, contexts and host threads: no grid's launch may depend on what ran before it.

  * FP64 lines four to a block whose staged window is just below 48 KB: with the kernel's
    static arrays they are above it, in a process that launched nothing larger before;
  * host threads with grids of their own at the same time.
"""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# windows of 1413 .. 1489 positions, four lines a block: y-lines with mu-hat, x-lines with
# the density, both force directions, and the window with mirrored halos between walls
FORCE_STAGES = [(600, 1413, False), (600, 1440, False), (1480, 600, False),
                (1480, 1480, False), (600, 1250, True)]


def check_force_stage(nx, ny, walls):
    from oracle import thermo
    from paper_1906_09530_gb300 import workloads as W
    from tests import cases
    rg, rl = thermo.maxwell(0.6)
    rho = W.with_noise(W.drop(nx, ny, rg, rl, 0.3 * min(nx, ny), 4.0), 7, 1e-4)
    c = dict(nx=nx, ny=ny, T_r=0.6, kappa=0.1, tau=0.9, k=0.5, order=6)
    g = cases.gpu_sim(c, walls_y=walls)
    g.set_fields(rho)
    got = g.fields()
    g.step(1)
    g.close()
    o = cases.oracle_sim(c, walls_y=walls)
    o.set_fields(rho)
    # (the bound of the other FP64 force stages, tests/test_gpu_lines64.py)
    for a, b in zip(got, o.fields()[:4]):
        assert np.abs(a - b).max() <= 1e-12 * max(np.abs(b).max(), 1e-3)


@pytest.mark.parametrize("nx,ny,walls", FORCE_STAGES)
def test_first_launch_of_a_process(cuda, nx, ny, walls):
    code = f"from tests.test_gpu_launch_limits import check_force_stage as c; c({nx}, {ny}, {walls})"
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


# 303 lines take two a block and 601 four, both with a ragged last group
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("lines", [303, 601])
@pytest.mark.parametrize("n", [1412, 1413, 1475, 1489, 1490, 1600, 1601])
def test_long_lines_side_by_side(cuda, n, lines, axis):
    """Tolerance 1e-13 of the largest derivative, as for single lines."""
    from oracle import cfd_alpha, cfd_line
    from paper_1906_09530_gb300 import lbm_cfd
    rng = np.random.default_rng(n + lines)
    u = rng.standard_normal((lines, n)) + 3.0
    v = u if axis == 0 else np.ascontiguousarray(u.T)
    d1, d2 = (d.cpu().numpy() for d in lbm_cfd(cuda.from_numpy(v).cuda(), axis, 6, True))
    if axis == 1:
        d1, d2 = d1.T, d2.T
    r1 = np.stack([cfd_line(x, cfd_alpha(6)) for x in u])
    r2 = np.stack([cfd_line(x, cfd_alpha(6)) for x in r1])
    assert np.abs(d1 - r1).max() <= 1e-13 * np.abs(r1).max()
    assert np.abs(d2 - r2).max() <= 1e-13 * np.abs(r2).max()


# (the sizes of one kernel's blocks, by grid: FP64 lines of 1600 and 1520 positions 52 832 and
# 50 176 bytes, double-float lines of 1000 and 64 positions 69 632 and 58 112, FP32 density
# lines of 52 and 128 positions 53 248 and 49 824)
@pytest.mark.parametrize("kind", ["fp64", "double-float", "fp32"])
def test_threads_with_different_grids(cuda, kind):
    """Two threads launch one kernel with block sizes of their own, each on its own stream:
    neither may lower the limit that the other's launch needs."""
    from paper_1906_09530_gb300 import Simulation, lbm_maxwell, lib
    torch = cuda
    rg, rl = lbm_maxwell(0.6)

    def work(size):
        s = torch.cuda.Stream()
        if kind == "fp32":
            sim = Simulation(size, size, 0.6, 0.1, 1.0, 0.5, precision="mixed", stream=s)
            rho = torch.full((size, size), rl, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            return lambda: lib().lbm_set_fields_device(sim.ctx, rho.data_ptr(), None, None)
        lines = 600 if kind == "fp64" else 64
        t = torch.float64 if kind == "fp64" else torch.float32
        u = [torch.ones((lines, size), dtype=t, device="cuda") for _ in range(4)]
        torch.cuda.synchronize()
        p = [x.data_ptr() for x in u]

        def call(_keep=u):
            if kind == "fp64":
                return lib().lbm_cfd(p[0], p[1], p[2], size, lines, 0, 6, s.cuda_stream)
            return lib().lbm_cfd_df(p[0], p[1], p[2], p[3], size, lines, 0, 6, s.cuda_stream)
        return call

    calls = [work(n) for n in {"fp64": (1600, 1520), "double-float": (1000, 64),
                               "fp32": (52, 128)}[kind]]
    bad = [0, 0]

    def loop(i):
        for k in range(4000):
            bad[i] += calls[i]() != 0

    threads = [threading.Thread(target=loop, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert bad == [0, 0]

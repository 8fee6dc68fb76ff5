"""Small grids of the mixed path: whole steps in one cluster launch give the bits of the same
steps launched pass by pass, and the chunked FP32 lines follow the oracle where their
geometry changes (few and many chunks, several windows, mirrored lines, odd rows)."""
import numpy as np
import pytest

from tests import cases

pytestmark = pytest.mark.gpu


def start(nx, ny, seed):
    from oracle import thermo
    from paper_1906_09530_gb300 import workloads as W
    rg, rl = thermo.maxwell(0.6)
    rho = W.flat(nx, ny, rg, rl, ny / 2, 6.0) if min(nx, ny) < 24 else \
        W.drop(nx, ny, rg, rl, 0.25 * min(nx, ny), 6.0)
    rho = W.with_noise(rho, seed, 1e-3)
    u = W.uniform_noise((ny, nx), seed + 1, 0.02)
    return rho, u, u[::-1].copy()


# one node above and below 8192, the largest grid; fewer rows than CTAs; rows that divide
# unevenly among them; the mu cap acting for the first steps only; 513 steps: two launches
@pytest.mark.parametrize("nx,ny,order,coll,steps", [
    (8, 8, 6, "bgk", 5), (8, 400, 6, "bgk", 513), (37, 29, 4, "mrt", 6), (64, 128, 6, "bgk", 4),
    (1024, 8, 4, "bgk", 3), (90, 91, 6, "mrt", 3), (331, 24, 6, "bgk", 3), (8193, 8, 6, "bgk", 2)])
def test_one_launch_equals_separate_passes(cuda, nx, ny, order, coll, steps):
    from paper_1906_09530_gb300 import Simulation
    got = []
    for timed in (False, True):
        s = Simulation(nx, ny, 0.6, 0.1, 1.1, 0.4, fd_order=order, precision="mixed",
                       collision=coll, mu_max=-0.02, mu_cap_steps=2)
        s.set_fields(*start(nx, ny, 5))
        if timed:
            for _ in range(steps):
                s.step_timed()
        else:
            s.step(steps - 2)
            s.step(2)
        assert s.t == steps
        got.append((s.get_populations()[0], *s.fields()))
        s.close()
    for a, b in zip(*got):
        assert np.isfinite(a).all() and np.array_equal(a, b)


def test_one_launch_reports_the_failing_step(cuda):
    """A density driven through the EOS pole is flagged at the same time level either way."""
    from paper_1906_09530_gb300 import LbmError, Simulation
    failed = []
    for timed in (False, True):
        s = Simulation(32, 32, 0.6, 0.1, 0.51, 1.0, precision="mixed")
        y, x = np.mgrid[0:32, 0:32]
        rho = 0.45 + 0.2 * np.cos(2 * np.pi * x / 32)
        with pytest.raises(LbmError):
            s.set_fields(rho, 0.3 * np.sin(2 * np.pi * x / 32))
            for _ in range(400):
                s.step_timed() if timed else s.step(1)
            s.step(1)
        failed.append(s.failed_step)
        s.close()
    assert failed[0] == failed[1] >= 0


@pytest.mark.parametrize("nx,ny,order,walls", [
    (100, 90, 6, False),      # 12 chunks a line
    (612, 300, 4, False),     # two windows, periods shorter than one
    (1500, 333, 6, False),    # three x windows
    (333, 1130, 6, False),    # odd rows, three y windows
    (444, 97, 6, True),       # mirrored lines shorter than a window
    (260, 900, 4, True)])     # and longer
def test_chunked_lines_follow_the_oracle(cuda, nx, ny, order, walls):
    from paper_1906_09530_gb300 import Simulation
    rho, ux, uy = start(nx, ny, 9)
    if walls:
        ux, uy = 0 * ux, 0 * uy
    s = Simulation(nx, ny, 0.6, 0.1, 1.0, 0.4, fd_order=order, precision="mixed", walls_y=walls)
    s.set_fields(rho, ux, uy)
    mu = s.fields()[3]
    s.step(20)
    r = s.fields()[0]
    s.close()
    o = cases.oracle_sim(dict(nx=nx, ny=ny, T_r=0.6, kappa=0.1, tau=1.0, k=0.4, order=order),
                         walls_y=walls)
    o.set_fields(rho, ux, uy)
    omu = o.fields()[3]
    # second derivatives of the noise, each FP32 sum over some ten terms of size rho_l
    assert np.abs(mu - omu).max() <= 1e-5 * max(np.abs(omu).max(), 0.1)
    o.step(20)
    assert cases.rel_err(r, o.fields()[0]) <= 1e-4

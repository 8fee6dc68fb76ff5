"""FP32 lines in full windows (grids above 2^19 nodes, and batches that want them): the bits of the chunked kernels on the same lines, and the oracle's derivatives where
their geometry changes (rows that are not whole 16-byte pieces, a ragged last line group, one
window on one axis and many on the other, mirrored lines)."""
import numpy as np
import pytest

from tests import cases

pytestmark = pytest.mark.gpu


def start(nx, ny, seed):
    from oracle import thermo
    from paper_1906_09530_gb300 import workloads as W
    rg, rl = thermo.maxwell(0.6)
    if min(nx, ny) > 100:
        rho = W.drop(nx, ny, rg, rl, 0.25 * min(nx, ny), 8.0)
    else:
        rho = W.flat(nx, ny, rg, rl, ny / 2, 8.0)
    return W.with_noise(rho, seed, 1e-3)


@pytest.mark.parametrize("order", [4, 6])
@pytest.mark.parametrize("nl", [8, 16])
@pytest.mark.parametrize("sizes", [
    [(1001, 600), (8, 400), (37, 29), (128, 96), (300, 700)],  # a large member
    [(64, 64), (8, 400), (300, 132)],                          # about one round of blocks
    [(512, 504)] * 10,                                         # most chunks needed
    [(256, 244)] * 20 + [(37, 29)]])                           # none of these: by pairs
def test_batch_in_full_windows(cuda, sizes, nl, order):
    """Batch members are solved in full windows or by (line, chunk) pairs as the whole batch
    wants it, a lone grid as it wants, or in one cluster launch: bit for bit the same."""
    from paper_1906_09530_gb300 import Batch, Simulation
    kw = dict(T_r=0.6, kappa=0.1, tau=1.0, k=0.4)
    rhos = [start(nx, ny, 3 + i) for i, (nx, ny) in enumerate(sizes)]
    b = Batch([dict(nx=nx, ny=ny, **kw) for nx, ny in sizes], fd_order=order)
    b.set_lines_per_block(nl)
    for i, r in enumerate(rhos):
        b.set_fields(i, r)
    b.step(5)
    for i, (nx, ny) in list(enumerate(sizes))[:5]:
        s = Simulation(nx, ny, 0.6, 0.1, 1.0, 0.4, fd_order=order, precision="mixed")
        s.set_fields(rhos[i])
        s.step(5)
        for name, x, y in zip(("rho", "vx", "vy", "mu"), b.fields(i), s.fields()):
            assert np.isfinite(x).all() and np.array_equal(x, y), (nx, ny, name)
        s.close()
    b.close()


@pytest.mark.parametrize("nx,ny,order,walls", [
    (1001, 603, 6, False),     # odd rows, 16 lines a block, two windows each way
    (2051, 1031, 4, False),    # odd rows, 8 lines a block
    (16, 140000, 6, False),    # one x window, 250 y windows: the order of tiles
    (140000, 16, 6, False),
    (901, 701, 4, True),       # mirrored lines with two windows
    (2500, 1000, 6, True)])
def test_large_grids_follow_the_oracle(cuda, nx, ny, order, walls):
    from paper_1906_09530_gb300 import Simulation
    rho = start(nx, ny, 9)
    s = Simulation(nx, ny, 0.6, 0.1, 1.0, 0.4, fd_order=order, precision="mixed", walls_y=walls)
    s.set_fields(rho)
    mu = s.fields()[3]
    s.step(2)
    r = s.fields()[0]
    s.close()
    o = cases.oracle_sim(dict(nx=nx, ny=ny, T_r=0.6, kappa=0.1, tau=1.0, k=0.4, order=order),
                         walls_y=walls)
    o.set_fields(rho)
    omu = o.fields()[3]
    # the bounds of the chunked lines (tests/test_gpu_small_grids.py)
    assert np.abs(mu - omu).max() <= 1e-5 * max(np.abs(omu).max(), 0.1)
    o.step(2)
    assert cases.rel_err(r, o.fields()[0]) <= 1e-4

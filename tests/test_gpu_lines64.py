"""The FP64 line solves where their chunking can go wrong: lines shorter than a warp, chunks
of 1 and 2 positions, remainders, lines cut into windows, the mirrored lines of walls below
and above one halo, 1, 2 and 4 lines a block; and the FP64 math of the EOS over its range.

References: the oracle's Thomas solve, and the oracle's force stage.  Tolerance 1e-13 of the
largest derivative, as for every other FP64 line solve (a few hundred roundings of 1e-16)."""
import numpy as np
import pytest

from tests import cases

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [4, 6])
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 31, 32, 33, 56, 63, 65, 255, 1000, 1600, 1601, 1793,
                               6144, 6145, 12100])
def test_lines_of_every_chunking(cuda, order, axis, n):
    from oracle import cfd_alpha, cfd_line
    from paper_1906_09530_gb300 import lbm_cfd
    rng = np.random.default_rng(n + order)
    u = rng.standard_normal((3, n)) + 3.0
    v = u if axis == 0 else np.ascontiguousarray(u.T)
    d1, d2 = (d.cpu().numpy() for d in lbm_cfd(cuda.from_numpy(v).cuda(), axis, order, True))
    if axis == 1:
        d1, d2 = d1.T, d2.T
    if n < 5:  # the symbol: the oracle's solve wants five positions
        th = 2 * np.pi * np.fft.fftfreq(n)
        al = cfd_alpha(order)
        sym = 1j * (2 / 3 * (al + 2) * np.sin(th) + (4 * al - 1) / 6 * np.sin(2 * th)) / (
            1 + 2 * al * np.cos(th))
        D = lambda w: np.fft.ifft(np.fft.fft(w, axis=1) * sym, axis=1).real  # noqa: E731
    else:
        D = lambda w: np.stack([cfd_line(x, cfd_alpha(order)) for x in w])  # noqa: E731
    r1 = D(u)
    r2 = D(r1)
    assert np.abs(d1 - r1).max() <= 1e-13 * max(np.abs(r1).max(), 1.0)
    assert np.abs(d2 - r2).max() <= 1e-13 * max(np.abs(r2).max(), 1.0)


@pytest.mark.parametrize("nx,ny", [(8, 8), (40, 31), (24, 192), (24, 193), (310, 300), (700, 40),
                                   (16, 1408), (16, 1409)])
def test_walled_force_stage(cuda, nx, ny):
    """The mirrored lines: whole periods up to 192 rows, one window with a halo above, windows
    above 1408; 310 and 700 columns take 2 and 4 lines a block."""
    from oracle import thermo
    from paper_1906_09530_gb300 import workloads as W
    rg, rl = thermo.maxwell(0.6)
    rho = W.with_noise(W.drop(nx, ny, rg, rl, 0.3 * min(nx, ny), 4.0), 7, 1e-4)
    c = dict(nx=nx, ny=ny, T_r=0.6, kappa=0.1, tau=0.9, k=0.5, order=6)
    g = cases.gpu_sim(c, walls_y=True)
    g.set_fields(rho)
    got = g.fields()
    g.step(3)
    got3 = g.fields()
    g.close()
    o = cases.oracle_sim(c, walls_y=True)
    o.set_fields(rho)
    for want in (o.fields()[:4],):
        for a, b in zip(got, want):
            assert np.abs(a - b).max() <= 1e-12 * max(np.abs(b).max(), 1e-3)
    o.step(3)
    for a, b in zip(got3, o.fields()[:4]):
        assert np.abs(a - b).max() <= 1e-11 * max(np.abs(b).max(), 1e-3)


def test_chemical_potential_over_twelve_decades(cuda):
    """mu-hat of uniform densities (no gradient): the FP64 logarithm and quotient against
    numpy's, from 1e-12 to the liquid, values around 1 included; to 8 units of the largest
    term."""
    from paper_1906_09530_gb300 import Simulation, make_eos, lbm_critical
    for kind, top in (("cs", 0.6), ("vdw", 9.5)):
        eos = make_eos(kind)
        T = 0.7 * lbm_critical(eos)[0]
        sim = Simulation(8, 8, 0.7, 0.1, 1.0, 1.0, precision="fp64", eos=eos)
        for r in np.r_[np.geomspace(1e-12, top, 60), np.linspace(0.9, 1.1, 21) * min(top, 1.0)]:
            sim.set_fields(np.full((8, 8), r))
            rho, _, _, mu = sim.fields()
            x = rho[0, 0]
            if kind == "cs":
                terms = [T * (3 - x) / (1 - x) ** 3, T * np.log(x), T, -2 * x]
            else:
                b, a = 2 / 21, 9 / 49
                terms = [T * np.log(x / (1 - b * x)), T / (1 - b * x), -2 * a * x]
            tol = 8 * 2.0**-53 * np.abs(terms).max()
            assert np.all(np.abs(mu - sum(terms)) <= tol), (kind, r)
        sim.close()


# 228 lines are the most that count as few, solved whole up to 1292 positions; 76 and 50 have
# room for two and three windows of 512, from 1025 positions on
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("n,lines", [(n, m) for n in (1292, 1293, 1599) for m in (228, 229)] +
                         [(1024, 76), (1025, 50), (1025, 51), (1536, 50), (1537, 50), (3001, 8)])
def test_few_lines_in_windows(cuda, n, lines, axis):
    """Tolerance 1e-13 of the largest derivative, as for single lines."""
    from oracle import cfd_alpha, cfd_line
    from paper_1906_09530_gb300 import lbm_cfd
    u = np.random.default_rng(n).standard_normal((lines, n)) + 3.0
    v = u if axis == 0 else np.ascontiguousarray(u.T)
    d1, d2 = (d.cpu().numpy() for d in lbm_cfd(cuda.from_numpy(v).cuda(), axis, 6, True))
    if axis == 1:
        d1, d2 = d1.T, d2.T
    r1 = np.stack([cfd_line(x, cfd_alpha(6)) for x in u])
    r2 = np.stack([cfd_line(x, cfd_alpha(6)) for x in r1])
    assert np.abs(d1 - r1).max() <= 1e-13 * np.abs(r1).max()
    assert np.abs(d2 - r2).max() <= 1e-13 * np.abs(r2).max()

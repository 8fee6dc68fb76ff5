"""Densities far from one: the gas of low reduced temperatures (2.9e-110 at T_r 0.03, 1.5e-173
at 0.02 in FP64), and units in which b is not of order one.  Nothing in the read-out or the
collision may leave the range of its type where the values themselves are in it.

Populations are multiples of 2^-12 of a scale 2^k, antisymmetric about a uniform density: the
sums are exact, the force is zero, and every result is the one at scale 1 (times 2^k)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def populations(nx, ny, k):
    rng = np.random.default_rng(nx)
    f = np.full((9, ny, nx), 0.0625)
    f[0] = 0.3125 - 5 * 2.0**-14
    for i, j in ((1, 3), (2, 4), (5, 7), (6, 8)):
        d = rng.integers(-200, 201, (ny, nx)) * 2.0**-12
        f[i] += d
        f[j] -= d
    return np.ldexp(f, k)


def simulation(nx, ny, k, precision, **kw):
    from paper_1906_09530_gb300 import Simulation, cs_eos
    eos = cs_eos(a=2.0**-k, b=4 * 2.0**-k) if k > 0 else None
    return Simulation(nx, ny, 0.6, 0.1, 1.0, 0.5, precision=precision, eos=eos, **kw)


@pytest.mark.parametrize("precision,k", [
    ("mixed", 88), ("mixed", 10), ("mixed", -50), ("mixed", -62), ("mixed", -100),
    ("mixed", -120), ("mixed", -132),
    ("fp64", 88), ("fp64", -99), ("fp64", -101), ("fp64", -600), ("fp64", -1040)])
def test_velocity_is_the_quotient(cuda, precision, k):
    """v = j / rho of the read-out and the diagnostics to one unit of FP64."""
    nx, ny = 37, 29
    f = populations(nx, ny, k)
    sim = simulation(nx, ny, k, precision)
    sim.set_populations(f)
    rho, vx, vy, _ = sim.fields()
    mass, vmax, rmin, rmax = sim.diag()
    sim.close()
    r = f.sum(axis=0)
    wx = ((f[1] + f[5] + f[8]) - (f[3] + f[6] + f[7])) / r
    wy = ((f[2] + f[5] + f[6]) - (f[4] + f[7] + f[8])) / r
    assert np.array_equal(rho, r)
    for v, w in ((vx, wx), (vy, wy)):
        assert np.all(np.abs(v - w) <= np.spacing(np.abs(w)))
    assert abs(vmax - np.sqrt(wx**2 + wy**2).max()) <= 4 * np.spacing(vmax)
    assert rmin == rmax == r[0, 0] and abs(mass - r.sum()) <= 1e-12 * mass


@pytest.mark.parametrize("collision", ["bgk", "mrt"])
@pytest.mark.parametrize("k", [-300, -600, -900])
def test_collision_at_any_scale(cuda, collision, k):
    """A uniform flow relaxes alike at every density: one step of the FP64 path, to 16 units
    of the largest population (the collision has some 60 roundings, most of smaller terms).
    Its terms u u rho are of size 0.01 rho here, not of (u rho)^2, which has no place in the
    type."""
    def stepped(k):
        f = np.repeat(np.repeat(populations(1, 1, 0), 16, 1), 16, 2)
        sim = simulation(16, 16, 0, "fp64", collision=collision)
        sim.set_populations(np.ldexp(f, k))
        sim.step(1)
        out = sim.get_populations()[0]
        sim.close()
        return np.ldexp(out, -k)

    want, got = stepped(0), stepped(k)
    assert np.abs(got - want).max() <= 16 * 2.0**-53 * want.max()


@pytest.mark.parametrize("precision", ["mixed", "mixed_df", "fp64"])
@pytest.mark.parametrize("k,node", [(0, 0.0), (-100, 0.0), (-100, np.nan), (0, np.nan)])
def test_velocity_without_a_value_is_nan(cuda, precision, k, node):
    """A node without a density makes the state unstable, which the next check says; what is
    read on the device before it has no velocity at that node, and not a number that looks
    like one."""
    from paper_1906_09530_gb300 import LbmError
    rho = np.full((29, 37), 2.0**k)
    rho[11, 17] = node
    sim = simulation(37, 29, k, precision)
    sim.set_fields_device(cuda.from_numpy(rho).cuda())
    _, vx, vy, _ = (a.cpu().numpy() for a in sim.fields_device())
    assert np.isnan(vx[11, 17]) and np.isnan(vy[11, 17])
    with pytest.raises(LbmError):
        sim.check()
    sim.close()

"""Readings of states beyond ordinary numbers: velocities where rho or the
momentum overflows, and crossings where the populations are far larger than
phi."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbf():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_0812_1282_gb300 as m

    return m


def rest(ny, nx):
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    return w * np.ones((9, ny, nx))


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_velocity_at_infinite_density(lbf, precision):
    """j / rho is 0 for a finite j and infinite rho, and the count of such
    nodes is of both components alike."""
    nx, ny = 37, 9
    f = rest(ny, nx)
    f[1, 4, 5] += 0.25
    f[3, 4, 5] += 0.125
    f[0, 4, 5] = np.inf
    f[0, 2, 3] = -np.inf
    sim = lbf.Lattice(lbf.params(precision=precision), nx, ny)
    sim.set_populations(f, np.zeros_like(f))
    rho, phi, ux, uy, st = sim.moments()
    assert st["nonfinite"] == 2
    assert rho[4, 5] == np.inf and rho[2, 3] == -np.inf
    assert ux[4, 5] == 0.0 and uy[4, 5] == 0.0 and ux[2, 3] == 0.0 and uy[2, 3] == 0.0
    f[0, 4, 5] = 4 / 9
    f[0, 2, 3] = 4 / 9 - 1.0  # rho = 0 exactly (f is stored less its rest value)
    f[1, 4, 5] = np.inf  # j and rho infinite: no number
    sim.set_populations(f, np.zeros_like(f))
    rho, phi, ux, uy, st = sim.moments()
    assert np.isnan(ux[4, 5]) and uy[4, 5] == 0.0
    assert rho[2, 3] == 0.0 and np.isnan(ux[2, 3]) and np.isnan(uy[2, 3])  # 0 / 0
    f[1, 2, 3], f[0, 2, 3] = 1 / 9 + 0.25, 4 / 9 - 1.25
    sim.set_populations(f, np.zeros_like(f))
    rho, phi, ux, uy, st = sim.moments()
    assert rho[2, 3] == 0.0 and ux[2, 3] == np.inf and np.isnan(uy[2, 3])
    sim.close()


def test_velocity_that_overflows(lbf):
    """rho = 0.7 and |j| = 1.6e308: u is infinite, with j's sign."""
    nx, ny = 33, 5
    f = rest(ny, nx)
    # summed in pairs (f0 + f1) + (f2 + f3), ...: +-8e307 cancel exactly
    f[1, 3, 7], f[2, 3, 7] = 8e307, -8e307
    f[3, 1, 9], f[4, 1, 9] = -8e307, 8e307
    f[8, 3, 7] -= 0.3
    f[8, 1, 9] -= 0.3
    sim = lbf.Lattice(lbf.params(precision="fp64"), nx, ny)
    sim.set_populations(f, np.zeros_like(f))
    rho, phi, ux, uy, st = sim.moments()
    assert 0.0 < rho[3, 7] < 0.95 and 0.0 < rho[1, 9] < 0.95
    for u, want in ((ux[3, 7], 1.6e308), (uy[1, 9], -1.6e308)):
        with np.errstate(over="ignore"):
            r = rho[3, 7] if want > 0 else rho[1, 9]
            assert u == np.float64(want) / r
    sim.close()


def crossings(phi):
    """The phi = 0 points on horizontal (periodic) and vertical links."""
    ny, nx = phi.shape
    pts = []
    for y in range(ny):
        for x in range(nx):
            a, b = phi[y, x], phi[y, (x + 1) % nx]
            if a * b < 0:
                pts.append((x + a / (a - b), y))
            if y + 1 < ny and a * phi[y + 1, x] < 0:
                pts.append((x, y + a / (a - phi[y + 1, x])))
    return pts


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("big", [2.0 ** 25, 2.0 ** 40])
def test_crossings_among_large_populations(lbf, oracle_mod, precision, big):
    """phi = -0.4 in a disc where g_1 = -g_3 = big, so that the sum of the g in
    FP32 comes out at about +0.5: the disc's edge is an interface."""
    nx, ny = 64, 48
    y, x = np.mgrid[0:ny, 0:nx]
    disc = np.hypot(x - 30.3, y - 20.2) < 11.4
    g = np.zeros((9, ny, nx))
    g[0] = np.where(disc, -0.9, 0.5)
    g[5] = np.where(disc, 0.5, 0.0)
    g[1] = np.where(disc, big, 0.0)
    g[3] = np.where(disc, -big, 0.0)
    sim = lbf.Lattice(lbf.params(precision=precision), nx, ny)
    sim.set_populations(rest(ny, nx), g)
    gs = sim.populations()[1]
    # in the order the library sums in FP64: pairs
    phi = (((gs[0] + gs[1]) + (gs[2] + gs[3])) + ((gs[4] + gs[5]) + (gs[6] + gs[7]))) + gs[8]
    assert (phi[disc] < 0).all() and (phi[~disc] > 0).all()
    assert len(crossings(phi)) > 40
    got = sim.contact_angle(exclude=0.0)
    want = oracle_mod.contact_angle(phi, exclude=0.0)
    for a, b in zip(got, want):
        assert abs(a - b) <= 1e-9 * max(1.0, abs(b))
    sim.close()

"""Readings of states beyond ordinary numbers: velocities where rho or the
momentum overflows."""
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

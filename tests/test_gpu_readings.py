"""Readings of a state: fields, statistics and the contact angle against
numpy on the populations read back.

Tolerances: fields are a dozen roundings of the storage type (FP64 4e-15, FP32
5e-7, relative to values of order 1); sums over n nodes n times that at most,
taken as n * 1e-15 (FP64) and n * 1e-7 (FP32) absolute.  The angle comes from
the phi points in FP64 on both sides."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

E = np.array([(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (-1, -1), (-1, 1), (1, -1)])


@pytest.fixture(scope="module")
def lbf():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_0812_1282_gb300 as m

    return m


def state(lbf, precision, nx, ny, seed):
    rng = np.random.default_rng(seed)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    f = w * (1 + 0.05 * rng.uniform(-1, 1, (9, ny, nx)))
    g = 0.1 * rng.uniform(-1, 1, (9, ny, nx))
    sim = lbf.Lattice(lbf.params(precision=precision), nx, ny)
    sim.set_populations(f, g)
    return sim


@pytest.mark.parametrize("precision,tol,per_node", [("fp64", 4e-15, 1e-15), ("fp32", 5e-7, 1e-7)])
@pytest.mark.parametrize("nx,ny", [(3, 3), (257, 3), (31, 40), (1023, 1031)])
def test_fields_and_statistics(lbf, precision, tol, per_node, nx, ny):
    sim = state(lbf, precision, nx, ny, nx)
    f, g = sim.populations()
    rho, phi, ux, uy, st = sim.moments()
    j = np.tensordot(E.T, f, 1)
    assert np.abs(rho - f.sum(0)).max() <= tol and np.abs(phi - g.sum(0)).max() <= tol
    assert np.abs(ux - j[0] / f.sum(0)).max() <= tol and np.abs(uy - j[1] / f.sum(0)).max() <= tol
    n = nx * ny
    for key, want in (("mass", f.sum()), ("order", g.sum()), ("mom_x", j[0].sum()),
                      ("mom_y", j[1].sum())):
        assert abs(st[key] - want) <= n * per_node
    assert abs(st["max_u"] - np.hypot(ux, uy).max()) <= tol
    assert st["nonfinite"] == 0
    again = sim.stats()
    assert again == st  # the same alone and beside the fields, and repeated
    f[3, ny // 2, nx // 2] = np.nan
    f[0, 0, 0] = np.inf
    sim.set_populations(f, g)
    r = sim.moments()
    assert r[4]["nonfinite"] == 2
    keep = np.isfinite(f.sum(0))
    assert np.array_equal(r[0][keep], rho[keep]) and np.array_equal(r[2][keep], ux[keep])
    sim.close()


@pytest.mark.parametrize("storage", [dict(precision="fp64"), dict(precision="fp32"),
                                     dict(precision="fp32", compact_g=True)])
@pytest.mark.parametrize("amp", [1.0, 1e-2, 1e-4])
def test_contact_angle_points(lbf, oracle_mod, storage, amp):
    """The interface of a drop of any amplitude: the FP32 look for crossings
    must miss none."""
    nx, ny = 203, 91
    y, x = np.mgrid[0:ny, 0:nx]
    phi0 = amp * np.tanh((31.3 - np.hypot(x - 100.2, y - 3.1)) / 1.4)
    sim = lbf.Lattice(lbf.params(collision="mrt", tau_alpha=1.5, tau_beta=0.6, **storage), nx, ny)
    sim.init_phi(phi0)
    sim.step(3)
    got = sim.contact_angle()
    want = oracle_mod.contact_angle(sim.moments()[1])
    for a, b in zip(got, want):
        assert abs(a - b) <= 1e-7 * max(1.0, abs(b))
    sim.close()

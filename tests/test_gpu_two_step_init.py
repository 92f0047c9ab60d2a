"""A new initial state directly after two-step launches on a compact domain,
with nothing in between that would put the ghost columns back: bit for bit and
byte for byte the one-step schedule's, for each way of setting it, both buffers
as the current one, even and odd widths."""
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


def start(lbf, sim, kind, page_locked):
    nx, ny = sim.nx, sim.ny
    if kind == "random":
        sim.init_random(0.4, 9)
    elif kind == "drop":
        sim.init_drop(0.3 * min(nx, ny), 0.1 * nx, 0.5 * ny)
    else:
        import torch

        phi0 = np.random.default_rng(nx + ny).uniform(-0.9, 0.9, (ny, nx))
        if page_locked:
            phi0 = torch.from_numpy(phi0).pin_memory().numpy()
        sim.init_phi(phi0)


@pytest.mark.parametrize("nx,ny", [(8, 8), (33, 9), (130, 21), (243, 34), (1210, 701)])
@pytest.mark.parametrize("before", [2, 4, 7])
@pytest.mark.parametrize("kind,page_locked", [("random", False), ("drop", False), ("phi", False),
                                              ("phi", True)])
@pytest.mark.parametrize("walls", [True, False])
def test_new_state_after_two_step_launches(lbf, nx, ny, before, kind, page_locked, walls):
    p = lbf.params(collision="mrt", tau_alpha=1.5, tau_beta=0.6, precision="fp32", compact_g=True,
                   walls=walls, h_bottom=0.1, h_top=-0.07)
    out = []
    for spl in (1, 2):
        sim = lbf.Lattice(p, nx, ny)
        sim.set_schedule(lbf.schedule(64, 16, steps_per_launch=spl))
        sim.init_random(0.3, 3)
        sim.step(before)
        start(lbf, sim, kind, page_locked)
        fields = sim.populations()
        sim.step(6)
        after = sim.populations()
        start(lbf, sim, kind, page_locked)
        out.append((*fields, *after, sim.save_state()))
        sim.close()
    assert all(np.array_equal(a, b) for a, b in zip(out[0][:4], out[1][:4]))
    assert out[0][4] == out[1][4]


def test_as_created(lbf):
    """The schedule a large domain starts with."""
    p = lbf.params(precision="fp32", compact_g=True, collision="mrt")
    used, fresh = lbf.Lattice(p, 1211, 701), lbf.Lattice(p, 1211, 701)
    assert used.schedule()["steps_per_launch"] == 2
    used.init_random(0.1, 1)
    used.step(100)
    for sim in (used, fresh):
        sim.init_drop(150.0, 40.0, 300.0)
    for a, b in zip(used.populations(), fresh.populations()):
        assert np.array_equal(a, b)
    assert used.save_state() == fresh.save_state()
    used.close()
    fresh.close()

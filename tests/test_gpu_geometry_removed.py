"""Steps after an obstacle map is taken off go on from the state it left: the
obstacle step keeps no periodic ghost columns, the others read them.  Against a
handle that never had a map, given the same populations: 1e-12 in FP64 (setting
them rounds once), 2e-6 in FP32, the suite's bounds for a few steps."""
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


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 2e-6)])
@pytest.mark.parametrize("nx,ny", [(41, 30), (130, 64)])
@pytest.mark.parametrize("walls", [True, False])
@pytest.mark.parametrize("tile", [None, (64, 8)])
@pytest.mark.parametrize("before", [30, 31])
def test_steps_after_removal(lbf, precision, tol, nx, ny, walls, tile, before):
    p = lbf.params(collision="mrt", tau_alpha=1.5, tau_beta=0.6, precision=precision, walls=walls,
                   h_bottom=0.05)
    cls = np.zeros((ny, nx), np.uint8)
    cls[10:14, 18:24] = 1
    sim, ref = lbf.Lattice(p, nx, ny), lbf.Lattice(p, nx, ny)
    if tile:
        sim.set_tile(*tile)
    sim.set_geometry(cls, [0.0, -0.1])
    sim.init_random(0.8, 5)
    sim.step(before)
    sim.set_geometry(None, None)
    f0, g0 = sim.populations()
    ref.set_populations(f0, g0)
    sim.step(3)
    ref.step(3)
    for a, b in zip(sim.populations(), ref.populations()):
        assert np.abs(a - b).max() <= tol
    sim.close()
    ref.close()


def test_batch_domain(lbf):
    p = lbf.params(collision="mrt", precision="fp64", walls=False)
    sizes = [(41, 30), (50, 33)]
    sim = lbf.Batch([p] * 2, *zip(*sizes))
    cls = np.zeros((33, 50), np.uint8)
    cls[10:14, 18:24] = 1
    sim.set_geometry(cls, [0.0, -0.1], dom=1)
    for k in range(2):
        sim.init_random(0.8, 5 + k, dom=k)
    sim.step(21)
    sim.set_geometry(None, None, dom=1)
    refs = []
    for k, s in enumerate(sizes):
        ref = lbf.Lattice(p, *s)
        ref.set_populations(*sim.populations(dom=k))
        ref.step(3)
        refs.append(ref.populations())
        ref.close()
    sim.step(3)
    for k in range(2):
        for a, b in zip(sim.populations(dom=k), refs[k]):
            assert np.abs(a - b).max() <= 1e-12
    sim.close()

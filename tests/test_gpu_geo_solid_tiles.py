"""The persistent obstacle step on maps with tiles of solid nodes only, which do
nothing and keep nobody waiting: the bits of a launch per step, over graphs of
every length and the single step, short last tiles too."""
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


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nx,ny,walls", [(200, 56, True), (161, 61, True), (131, 43, False)])
def test_solid_tiles(lbf, precision, nx, ny, walls):
    cls = np.zeros((ny, nx), np.uint8)
    cls[:, nx // 4:] = 2  # columns of whole solid tiles beside a channel
    cls[ny // 2 - 4:ny // 2 + 5, nx // 4:] = 0
    p = lbf.params(collision="mrt", tau_alpha=1.5, tau_beta=0.6, precision=precision, walls=walls,
                   h_bottom=0.05)
    phi0 = np.random.default_rng(nx).uniform(-0.8, 0.8, (ny, nx))
    phi0[cls != 0] = 0.0
    out = []
    for persist in (0, 1):
        sim = lbf.Lattice(p, nx, ny)
        sim.set_geometry(cls, [0.0, -0.1, 0.08])
        sim.set_schedule(lbf.schedule(128, 16, ctas_per_sm=0, persist=persist))
        sim.init_phi(phi0)
        for n in (1, 64, 7, 7, 130, 2):
            sim.step(n)
        sim.sync()
        out.append(sim.populations())
        sim.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])

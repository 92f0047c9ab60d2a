"""The obstacle step's tile list: domains of many tiles (4-row tiles in
FP32), tiles without a solid neighbour, short last tiles, tiles of solid
nodes only.  Against the oracle after 6 steps (FP64 1e-13: about 6 x 2 x 150
roundings of numbers of order 1; FP32 2e-6, the suite's bound for a few
steps), and bit for bit against the two-step form, whose tiles are fixed."""
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


def block_map(nx, ny, walls):
    cls = np.zeros((ny, nx), np.uint8)
    for k, (x, y) in enumerate([(9, 6), (30, 9), (nx // 2, 5), (nx - 12, ny - 9)]):
        cls[y:y + 3 + k % 2, x:x + 4] = 1 + k % 2
    cls[:, nx // 3:nx // 3 + 70] = 2  # whole tiles of solid nodes
    cls[ny // 2 - 3:ny // 2 + 3, nx // 3:nx // 3 + 70] = 0
    return cls


@pytest.mark.parametrize("nx,ny", [(1301, 131), (1101, 85), (333, 30), (227, 37)])
@pytest.mark.parametrize("walls", [True, False])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-13), ("fp32", 2e-6)])
def test_tile_list(lbf, oracle_mod, nx, ny, walls, precision, tol):
    kw = dict(collision="mrt", tau_alpha=1.5, tau_beta=0.6, h_bottom=0.05, h_top=-0.04, walls=walls)
    cls = block_map(nx, ny, walls)
    hc = [0.0, -0.1, 0.08]
    phi0 = np.random.default_rng(nx).uniform(-0.8, 0.8, (ny, nx))
    phi0[cls != 0] = 0.0
    ref = oracle_mod.OracleLattice(oracle_mod.params(**kw), nx, ny)
    ref.set_geometry(cls, hc)
    ref.init_phi(phi0)
    ref.step(6)
    out = []
    for spl in (1, 2):
        sim = lbf.Lattice(lbf.params(precision=precision, **kw), nx, ny)
        sim.set_geometry(cls, hc)
        sim.set_schedule(lbf.schedule(128, 16, steps_per_launch=spl))
        sim.init_phi(phi0)
        sim.step(6)
        out.append(sim.populations())
        sim.close()
    fl = cls == 0
    for k, want in ((0, ref.f), (1, ref.g)):
        assert np.abs(out[0][k][:, fl] - want[:, fl]).max() <= tol
        assert np.array_equal(out[0][k], out[1][k])

"""The FP64 step at the edges of its tiles (CTA-shared phi, halo columns,
running row values, wall ghost rows) against the oracle, and bit for bit
between launch shapes.

Tolerance: a step is about 120 roundings of numbers of order 1 or below on
either side, 2 x 20 x 120 x 2^-53 = 5.3e-13 over 20 steps of a stable scheme;
1e-12 is the suite's bound for FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-12
SIZES = [(3, 3), (31, 4), (32, 5), (33, 3), (65, 7), (130, 9)]
SHAPES = [(32, 1), (64, 2), (96, 3), (256, 4), (128, 32)]


@pytest.fixture(scope="module")
def lbf():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_0812_1282_gb300 as m

    return m


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("collision,relax,step2", [("bgk", False, False), ("bgk", False, True),
                                                   ("mrt", False, True), ("mrt", True, True)])
@pytest.mark.parametrize("walls,rule,tau_phi", [(True, 0, 1.0), (True, 1, 0.8), (False, 0, 0.8)])
def test_tile_edges_match_oracle(lbf, oracle_mod, nx, ny, collision, relax, step2, walls, rule, tau_phi):
    kw = dict(collision=collision, tau_alpha=1.5, tau_beta=0.6, tau_phi=tau_phi, h_bottom=-0.1,
              h_top=0.07, walls=walls, step2_relax_momentum=relax, zero_u_at_walls=step2,
              wetting_rule=rule)
    rng = np.random.default_rng(nx * 1000 + ny)
    phi0 = rng.uniform(-0.9, 0.9, (ny, nx))
    ref = oracle_mod.OracleLattice(oracle_mod.params(**kw), nx, ny)
    ref.init_phi(phi0)
    ref.step(20)
    first = None
    for bx, rows in SHAPES:
        sim = lbf.Lattice(lbf.params(precision="fp64", **kw), nx, ny)
        sim.set_tile(bx, rows)
        sim.init_phi(phi0)
        sim.step(20)
        f, g = sim.populations()
        sim.close()
        if first is None:
            first = (f, g)
            assert np.abs(f - ref.f).max() <= TOL
            assert np.abs(g - ref.g).max() <= TOL
        assert np.array_equal(f, first[0]) and np.array_equal(g, first[1])

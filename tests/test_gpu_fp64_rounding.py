"""A step of the FP64 forms rounds the order parameter once per node: g_0, which
carries it, advances by the difference of the other populations' sums, and those
are a hundred times smaller here.  So with phi between 1/2 and 1 the total changes
by sqrt(nodes) 2^-53 / sqrt(12) a step, rms over steps (a rounding of numbers in
[1/2, 1) is uniform in +-2^-54).  Bound: 1.5 times that, 3.5 standard deviations of
an rms over 24 steps.  The walls, the obstacles and the periodic edges conserve it
exactly."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

STEPS = 24


@pytest.fixture(scope="module")
def lbf():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_0812_1282_gb300 as m

    return m


def rms_change(sim, nodes, dom=0):
    """rms over steps of the change of the total of g, per sqrt(node)."""
    def g():
        return sim.populations(dom=dom)[1].ravel()

    sim.step(3)
    last, sq = g(), 0.0
    for _ in range(STEPS):
        sim.step(1)
        now = g()
        sq += math.fsum(np.concatenate([now, -last])) ** 2  # exact up to its last rounding
        last = now
    return math.sqrt(sq / STEPS / nodes)


def field(nx, ny):
    return np.random.default_rng(nx + ny).uniform(0.65, 0.85, (ny, nx))


BOUND = 1.5 * 2.0 ** -53 / math.sqrt(12.0)


# two threads per node, one, the staged step, and the obstacle step of few tiles and many
@pytest.mark.parametrize("nx,ny,tile,block", [(100, 50, None, False), (200, 100, None, False),
                                              (130, 64, (64, 8), False), (150, 60, None, True),
                                              (401, 150, None, True)])
@pytest.mark.parametrize("collision,walls,tau_phi", [("mrt", True, 1.0), ("bgk", False, 1.0),
                                                     ("mrt", False, 0.8)])
def test_one_rounding_a_step(lbf, nx, ny, tile, block, collision, walls, tau_phi):
    sim = lbf.Lattice(lbf.params(collision=collision, tau_alpha=1.5, tau_beta=0.6, tau_phi=tau_phi,
                                 precision="fp64", walls=walls), nx, ny)
    if tile:
        sim.set_tile(*tile)
    cls = np.zeros((ny, nx), np.uint8)
    if block:
        cls[20:30, 40:60] = 1
        sim.set_geometry(cls, [0.0, 0.0])
    sim.init_phi(np.where(cls, 0.0, field(nx, ny)))
    got = rms_change(sim, int((cls == 0).sum()))
    sim.close()
    assert got <= BOUND


def test_batch(lbf):
    sizes = [(64, 40), (150, 61)]
    sim = lbf.Batch([lbf.params(collision="mrt", tau_alpha=1.5, tau_beta=0.6, precision="fp64")] * 2,
                    *zip(*sizes))
    for k, (nx, ny) in enumerate(sizes):
        sim.init_phi(field(nx, ny), dom=k)
    got = rms_change(sim, 150 * 61, dom=1)
    sim.close()
    assert got <= BOUND

"""What a handle reports as its schedule is what it runs, counted in launches
per step."""
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


def params(lbf, storage, **kw):
    return lbf.params(collision="mrt", tau_alpha=1.5, tau_beta=0.6,
                      precision="fp64" if storage == "fp64" else "fp32",
                      compact_g=storage == "compact", **kw)


def launches(sim, n):
    """Launches of n steps, the graphs and ghost columns they need in place."""
    sim.step(n)
    sim.sync()
    before = sim.launch_count
    sim.step(n)
    return sim.launch_count - before


@pytest.mark.parametrize("block_x,rows,steps", [(64, 64, 2), (96, 64, 2), (128, 64, 2), (64, 16, 1),
                                                (32, 64, 1), (160, 64, 1), (256, 64, 1),
                                                (288, 120, 1)])
def test_tile_of_a_large_compact_domain(lbf, block_x, rows, steps):
    sim = lbf.Lattice(params(lbf, "compact"), 1210, 701)
    sim.set_tile(block_x, rows)
    assert sim.tile() == (block_x, rows)
    assert sim.schedule()["steps_per_launch"] == steps
    sim.init_random(0.1, 3)
    assert launches(sim, 64) == 64 // steps
    sim.close()

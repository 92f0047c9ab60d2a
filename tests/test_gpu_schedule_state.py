"""What a handle reports as its schedule is what it runs, and a schedule read
and set again or an autotuned obstacle map that is taken off leaves it on the
step it had: counted in launches per step."""
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


def as_schedule(lbf, d):
    return lbf.schedule(d["block_x"], d["rows"], ctas_per_sm=d["ctas_per_sm"], max_nx=d["max_nx"],
                        order=d["order"], chains=d["chains"], persist=d["persist"],
                        fill_pct=d["fill_pct"], seal_edges=d["seal_edges"],
                        steps_per_launch=d["steps_per_launch"])


@pytest.mark.parametrize("storage", ["fp32", "compact"])
def test_schedule_read_and_set_again(lbf, storage):
    """A small lattice keeps its step of several steps per launch; a shape
    that was set, the same one too, selects the general step."""
    sim = lbf.Lattice(params(lbf, storage), 120, 50)
    sim.init_random(0.1, 3)
    before = launches(sim, 64)
    assert before < 64
    sched = sim.schedule()
    sim.set_schedule(as_schedule(lbf, sched))
    assert sim.schedule() == sched
    assert launches(sim, 64) == before
    other = lbf.Lattice(params(lbf, storage), 120, 50)
    other.set_schedule(as_schedule(lbf, sched))  # a saved one, on a handle of the same lattice
    other.init_random(0.1, 3)
    assert launches(other, 64) == before
    sim.set_tile(*sim.tile())
    assert launches(sim, 64) == 64
    sim.set_schedule(as_schedule(lbf, sim.schedule()))
    assert launches(sim, 64) == 64
    other.set_schedule(lbf.schedule(64, 8))
    assert launches(other, 64) == 64
    other.set_schedule(as_schedule(lbf, sched))
    assert launches(other, 64) == before
    sim.close()
    other.close()


def test_batch_schedule_read_and_set_again(lbf):
    """A small batch likewise; its steps leave the same bytes."""
    sizes = [(33, 20), (64, 31), (90, 44)]
    out = []
    for again in (False, True):
        sim = lbf.Batch([params(lbf, "fp32")] * 3, *zip(*sizes))
        if again:
            sim.set_schedule(as_schedule(lbf, sim.schedule()))
        for k in range(3):
            sim.init_random(0.3, k, dom=k)
        sim.step(9)
        out.append((sim.save_state(), sim.schedule()))
        sim.close()
    assert out[0] == out[1]


def test_autotuned_with_obstacles_then_without(lbf):
    nx, ny = 120, 50
    sim = lbf.Lattice(params(lbf, "fp32"), nx, ny)
    sim.init_random(0.1, 3)
    before = launches(sim, 64)
    cls = np.zeros((ny, nx), np.uint8)
    cls[20:24, 30:36] = 1
    sim.set_geometry(cls, [0.0, 0.1])
    sim.init_random(0.1, 3)
    sim.autotune(reps=1)
    sim.set_geometry(None, None)
    sim.init_random(0.1, 3)
    assert launches(sim, 64) == before
    sim.close()

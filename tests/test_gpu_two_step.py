"""Two steps per launch on a single compact domain (lb_schedule
steps_per_launch = 2) against one step per launch, bit for bit and byte for
byte of the checkpoint: strips that end inside and at the domain's edge, tiles
of a few rows and of the whole domain, walls and periodic rows, odd step
counts, a new initial state and a loaded one in between."""
import os
import subprocess
import sys

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


def params(lbf, collision="mrt", **kw):
    return lbf.params(collision=collision, tau_alpha=1.5, tau_beta=0.6, precision="fp32",
                      compact_g=True, **kw)


def lattice(lbf, p, nx, ny, shape):
    sim = lbf.Lattice(p, nx, ny)
    if shape:
        sim.set_schedule(lbf.schedule(*shape, steps_per_launch=2))
    else:
        sim.set_schedule(lbf.schedule(64, 5, steps_per_launch=1))
    sim.init_random(0.3, 3)
    return sim


@pytest.mark.parametrize("nx,ny", [(8, 8), (33, 9), (118, 20), (119, 31), (242, 40), (243, 17),
                                   (500, 70)])
@pytest.mark.parametrize("collision,walls,rule", [("mrt", True, 0), ("mrt", True, 1),
                                                  ("mrt", False, 0), ("bgk", True, 0)])
def test_bits(lbf, nx, ny, collision, walls, rule):
    p = params(lbf, collision, walls=walls, wetting_rule=rule, h_bottom=0.1, h_top=-0.07,
               mrt_lut=7 if collision == "mrt" and rule else 0)
    ref = lattice(lbf, p, nx, ny, None)
    ref.step(21)
    want = ref.save_state()
    ref.close()
    for shape in ((64, 3), (64, 16), (96, 8), (128, 2), (128, 64)):
        sim = lattice(lbf, p, nx, ny, shape)
        sim.step(9)
        sim.step(12)
        assert sim.save_state() == want, shape
        sim.close()


def test_other_kernels_between(lbf):
    """Single steps, a set wetting gradient, another shape, a checkpoint and a
    new initial state between two-step launches."""
    nx, ny = 251, 60
    p = params(lbf)
    out = []
    for shape in (None, (64, 7)):
        sim = lattice(lbf, p, nx, ny, shape)
        sim.step(4)
        sim.step(1)
        sim.set_wetting(0.08, 0.0)
        sim.step(6)
        blob = sim.save_state()
        sim.step(130)
        sim.load_state(blob)
        sim.step(8)
        if shape:
            sim.set_schedule(lbf.schedule(128, 33, steps_per_launch=2))
        sim.step(5)
        a = sim.save_state()
        sim.init_random(0.2, 9)
        b = sim.save_state()
        sim.step(10)
        out.append((blob, a, b, sim.save_state(), *sim.populations()))
        sim.close()
    assert out[0][:4] == out[1][:4]
    assert all(np.array_equal(u, v) for u, v in zip(out[0][4:], out[1][4:]))


def test_large_domain_starts_with_it(lbf):
    nx, ny = 1210, 701
    p = params(lbf, h_bottom=0.05)
    a = lbf.Lattice(p, nx, ny)
    assert a.schedule()["steps_per_launch"] == 2
    b = lbf.Lattice(p, nx, ny)
    b.set_tile(64, 8)
    assert b.schedule()["steps_per_launch"] == 1
    for sim in (a, b):
        sim.init_random(0.3, 5)
        sim.step(13)
    assert a.save_state() == b.save_state()
    before = a.save_state()
    a.autotune(reps=1)
    assert a.save_state() == before
    a.step(7)
    b.step(7)
    assert a.save_state() == b.save_state()
    a.close()
    b.close()


def test_large_domain_starts_with_it_in_a_new_process(lbf):
    """The rule asks for the kernel's occupancy before any two-step schedule was
    set in the process."""
    code = ("import paper_0812_1282_gb300 as lbf\n"
            "p = lbf.params(precision='fp32', compact_g=True)\n"
            "assert lbf.Lattice(p, 1210, 701).schedule()['steps_per_launch'] == 2\n")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run([sys.executable, "-c", code], check=True, cwd=root, timeout=300)

"""The launch shape a handle starts with (chosen from its domains' sizes)
leaves results as any explicit one does, bit for bit: tiny and ragged
lattices, one wave of CTAs and several, each storage."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

STORAGE = {"fp64": dict(precision="fp64"), "fp32": dict(precision="fp32"),
           "compact": dict(precision="fp32", compact_g=True)}


@pytest.fixture(scope="module")
def lbf():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_0812_1282_gb300 as m

    return m


def run(lbf, plist, sizes, tile):
    sim = lbf.Batch(plist, *zip(*sizes)) if len(sizes) > 1 else lbf.Lattice(plist[0], *sizes[0])
    if tile:
        sim.set_tile(*tile)
    for k in range(len(sizes)):
        sim.init_random(0.3, 11 + k, dom=k)
    sim.step(7)
    out = [sim.populations(dom=k) for k in range(len(sizes))]
    sim.close()
    return out


@pytest.mark.parametrize("storage", sorted(STORAGE))
@pytest.mark.parametrize("sizes", [[(3, 3)], [(28, 15)], [(517, 3)], [(5, 701)], [(301, 97)],
                                   [(1301, 811)], [(33, 5), (250, 41), (3, 3)],
                                   [(190 + 7 * k, 130 + 3 * k) for k in range(24)]],
                         ids=lambda s: "-".join("%dx%d" % v for v in s[:2]))
@pytest.mark.parametrize("walls", [True, False])
def test_default_shape_is_bit_identical(lbf, storage, sizes, walls):
    p = lbf.params(collision="mrt", tau_alpha=1.5, tau_beta=0.6, walls=walls, h_bottom=0.05,
                   **STORAGE[storage])
    a = run(lbf, [p] * len(sizes), sizes, None)
    b = run(lbf, [p] * len(sizes), sizes, (64, 32))
    for (fa, ga), (fb, gb) in zip(a, b):
        assert np.array_equal(fa, fb) and np.array_equal(ga, gb)


@pytest.mark.parametrize("storage", sorted(STORAGE))
@pytest.mark.parametrize("nx,ny", [(3, 3), (4, 33), (31, 6), (33, 5), (66, 8), (131, 29),
                                   (131, 76), (203, 97)])
@pytest.mark.parametrize("walls,rule", [(True, 0), (True, 1), (False, 0)])
@pytest.mark.parametrize("collision,relax,lut,tau_phi", [("bgk", False, 0, 1.0), ("bgk", False, 0, 0.8),
                                                         ("mrt", False, 0, 1.0), ("mrt", True, 9, 1.0),
                                                         ("mrt", False, 0, 1.3)])
def test_small_lattice_step_is_bit_identical(lbf, storage, nx, ny, walls, rule, collision, relax,
                                             lut, tau_phi):
    """The step a small single domain starts with against the staged step,
    switching from one to the other on the way, ghost columns included."""
    if storage == "compact" and tau_phi != 1.0:
        pytest.skip("compact storage needs tau_phi = 1")
    p = lbf.params(collision=collision, tau_alpha=1.5, tau_beta=0.6, tau_phi=tau_phi, walls=walls,
                   wetting_rule=rule, h_bottom=0.1, h_top=-0.07, step2_relax_momentum=relax,
                   mrt_lut=lut, **STORAGE[storage])
    phi0 = np.random.default_rng(nx * 100 + ny).uniform(-0.9, 0.9, (ny, nx))
    out = []
    for first in (0, 9):
        sim = lbf.Lattice(p, nx, ny)
        sim.init_phi(phi0)
        sim.step(first)
        sim.set_tile(64, 2)
        sim.step(18 - first)
        out.append((*sim.populations(), sim.save_state()))
        sim.close()
    small = lbf.Lattice(p, nx, ny)
    small.init_phi(phi0)
    small.step(18)
    out.append((*small.populations(), small.save_state()))
    small.close()
    for f, g, blob in out[1:]:
        assert np.array_equal(f, out[0][0]) and np.array_equal(g, out[0][1])
        assert blob == out[0][2]


@pytest.mark.parametrize("storage", ["compact", "fp32"])
@pytest.mark.parametrize("nx,ny", [(7, 30), (30, 7), (8, 8), (9, 31), (20, 9), (41, 8), (131, 76), (203, 97),
                                   (215, 105), (245, 110), (320, 200)])
@pytest.mark.parametrize("collision,walls,rule,lut,tau_phi", [("bgk", True, 0, 0, 1.0),
                                                              ("mrt", True, 1, 9, 1.0),
                                                              ("mrt", False, 0, 0, 1.0),
                                                              ("bgk", False, 0, 0, 0.8)])
def test_several_steps_per_launch_are_bit_identical(lbf, storage, nx, ny, collision, walls, rule, lut,
                                                    tau_phi):
    """Small FP32 lattices, stepped by whole graphs, remainders and single steps
    with a change of the wetting in between, against the staged step: lattices
    narrower than a tile's border, of one tile, and of four, three and two steps
    per launch and two tiles per SM."""
    if storage == "compact" and tau_phi != 1.0:
        pytest.skip("compact storage needs tau_phi = 1")
    p = lbf.params(collision=collision, tau_alpha=1.5, tau_beta=0.6, tau_phi=tau_phi, walls=walls,
                   wetting_rule=rule, h_bottom=0.1, h_top=-0.07, mrt_lut=lut, **STORAGE[storage])
    out = []
    for staged in (True, False):
        sim = lbf.Lattice(p, nx, ny)
        if staged:
            sim.set_tile(64, 2)
        sim.init_random(0.3, nx + ny)
        for n in (64, 7, 1, 7, 2, 7, 66):
            sim.step(n)
            sim.set_wetting(0.1 - 0.001 * n, 0.05)
        out.append((*sim.populations(), sim.save_state()))
        sim.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2]


@pytest.mark.parametrize("storage", sorted(STORAGE))
@pytest.mark.parametrize("collision,relax,walls,tau_phi", [("bgk", False, True, 1.0),
                                                           ("mrt", True, True, 1.0),
                                                           ("mrt", False, False, 1.0),
                                                           ("bgk", False, False, 0.8),
                                                           ("mrt", False, True, 1.3)])
def test_small_batch_is_bit_identical(lbf, storage, collision, relax, walls, tau_phi):
    """The step a small batch starts with against the staged one, domain by
    domain with gradients of their own, and after a change of schedule and an
    autotuned one."""
    if storage == "compact" and tau_phi != 1.0:
        pytest.skip("compact storage needs tau_phi = 1")
    sizes = [(3, 3), (31, 6), (33, 5), (64, 4), (66, 29), (131, 8), (200, 61)]
    plist = [lbf.params(collision=collision, tau_alpha=1.5, tau_beta=0.6 + 0.02 * k, walls=walls,
                        tau_phi=tau_phi,
                        h_bottom=0.02 * k, h_top=-0.01 * k, step2_relax_momentum=relax,
                        **STORAGE[storage]) for k in range(len(sizes))]
    out = []
    for mode in ("staged", "small", "switch", "tuned"):
        sim = lbf.Batch(plist, *zip(*sizes))
        if mode == "staged":
            sim.set_tile(64, 7)
        for k in range(len(sizes)):
            sim.init_random(0.4, 3 + k, dom=k)
        if mode == "tuned":
            sim.autotune(reps=1)
        sim.step(9)
        if mode == "switch":
            sim.set_tile(96, 3)
        sim.set_wetting(0.06, 0.03, dom=4)
        sim.step(10)
        out.append(sim.save_state())
        sim.close()
    assert out[1:] == out[:1] * 3

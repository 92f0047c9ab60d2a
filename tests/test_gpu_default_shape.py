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

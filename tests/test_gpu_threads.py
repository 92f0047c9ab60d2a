"""Handles of several host threads side by side, whose launches of the same
kernel differ in the shared memory they ask for: none is refused, and each
leaves the bytes it leaves alone."""
import threading

import pytest

pytestmark = pytest.mark.gpu

SIZES = [(200, 100), (200, 75), (200, 60), (200, 50), (120, 40)]
HANDLES = 30  # per thread


@pytest.fixture(scope="module")
def lbf():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_0812_1282_gb300 as m

    return m


def steps(lbf, p, nx, ny, stream):
    sim = lbf.Lattice(p, nx, ny, stream=stream)
    try:
        sim.init_random(0.2, nx + ny)
        for n in (6, 6, 10, 10, 64):  # a graph of a remainder from its second time on
            sim.step(n)
        return sim.save_state()
    finally:
        sim.close()


@pytest.mark.parametrize("storage", [dict(compact_g=True), dict()], ids=["compact", "full"])
def test_small_lattices_of_several_threads(lbf, storage):
    import torch

    p = lbf.params(collision="mrt", tau_alpha=1.5, tau_beta=0.6, precision="fp32", **storage)
    alone = [steps(lbf, p, nx, ny, None) for nx, ny in SIZES]
    wrong = []

    def work(k):
        stream = torch.cuda.Stream()
        for _ in range(HANDLES):
            try:
                if steps(lbf, p, *SIZES[k], stream) != alone[k]:
                    wrong.append((SIZES[k], "other bytes"))
            except lbf.LBError as e:
                wrong.append((SIZES[k], str(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(SIZES))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, (len(wrong), wrong[:3])

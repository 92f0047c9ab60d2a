"""Which obstacle maps are accepted, against the rules node by node, on random
maps whose neighbourhoods wrap around the lattice."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
WALL = 8


@pytest.fixture(scope="module")
def lbf():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_0812_1282_gb300 as m

    return m


def accepted(cls, walls):
    ny, nx = cls.shape

    def at(x, y):
        return cls[y % ny, x % nx]

    def solid(x, y):
        return (walls and not 0 <= y < ny) or at(x, y) != 0

    for y in range(ny):
        for x in range(nx):
            if cls[y, x] == WALL and (not walls or y not in (0, ny - 1) or ny < 4
                                      or cls[y + (1 if y == 0 else -1), x] != 0):
                return False
    if not (cls == 0).any():
        return False
    for y in range(-1 if walls else 0, ny + 1 if walls else ny):
        for x in range(nx):
            if not solid(x, y) or at(x, min(max(y, 0), ny - 1)) == WALL and not 0 < y < ny - 1:
                continue
            axis = [d for d in ((1, 0), (-1, 0), (0, 1), (0, -1)) if not solid(x + d[0], y + d[1])]
            diag = [d for d in ((1, 1), (-1, -1), (-1, 1), (1, -1)) if not solid(x + d[0], y + d[1])]
            if any(solid(x + 2 * d[0], y + 2 * d[1]) for d in axis or diag):
                return False
    return True


@pytest.mark.parametrize("nx,ny", [(3, 3), (4, 5), (5, 4), (7, 6), (12, 9)])
@pytest.mark.parametrize("walls", [True, False])
def test_accepted_maps(lbf, nx, ny, walls):
    rng = np.random.default_rng(100 * nx + ny + walls)
    sim = lbf.Lattice(lbf.params(precision="fp32", walls=walls), nx, ny)
    seen = [0, 0]
    for k in range(300):
        cls = np.zeros((ny, nx), np.uint8)
        if k % 3 == 0:
            cls[rng.random((ny, nx)) < rng.choice([0.03, 0.3, 0.9])] = 1
        else:  # a block, across the edges too
            x0, y0, w, h = rng.integers(nx), rng.integers(ny), rng.integers(1, nx + 1), rng.integers(1, ny + 1)
            cls[np.ix_((y0 + np.arange(h)) % ny, (x0 + np.arange(w)) % nx)] = 2
        if k % 5 == 0:
            cls[0, rng.random(nx) < 0.5] = WALL
            cls[-1] = np.where(rng.random(nx) < 0.2, WALL, cls[-1])
        want = accepted(cls, walls)
        seen[want] += 1
        try:
            sim.set_geometry(cls, [0.0, 0.1, -0.1])
            got = True
        except lbf.LBError:
            got = False
        assert got == want, cls
    assert seen[0] > 20
    sim.close()

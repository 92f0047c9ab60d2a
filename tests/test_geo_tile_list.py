"""The obstacle step's tile list, made row by row, against its definition node by
node on random maps: which tiles hold a fluid or wall node, which of them fluid
with a solid neighbour, in order.  Host only."""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0812_1282_gb300", "csrc")
KNODEWALL = 8

MAIN = r"""
#include <cstdio>
#include <vector>
#include "lb_geo_persist.h"
int main()
{
    int precision, sm, nx, ny, walls;
    while (std::scanf("%d %d %d %d %d", &precision, &sm, &nx, &ny, &walls) == 5) {
        std::vector<unsigned char> cls(size_t(nx) * ny);
        for (auto& c : cls) {
            int v;
            if (std::scanf("%d", &v) != 1) return 1;
            c = static_cast<unsigned char>(v);
        }
        const lbfe::GeoTiles t = lbfe::make_geo_tiles(precision, sm, cls.data(), nx, ny, walls);
        std::printf("%d", t.rows);
        for (int v : t.list) std::printf(" %d", v);
        std::printf("\n");
    }
}
"""


def expected(precision, sm, cls, walls):
    ny, nx = cls.shape

    def tiles(ty):
        near, plain = [], []
        ntx = -(-nx // 32)
        for q in range(ntx * -(-ny // ty)):
            x0, y0 = q % ntx * 32, q // ntx * ty
            live = touches = False
            for y in range(y0, min(y0 + ty, ny)):
                for x in range(x0, min(x0 + 32, nx)):
                    live = live or cls[y, x] in (0, KNODEWALL)
                    if cls[y, x] != 0:
                        continue
                    for dy in (-1, 0, 1):
                        for dx in (-1, 0, 1):
                            out = walls and not 0 <= y + dy < ny
                            touches = touches or out or cls[(y + dy) % ny, (x + dx) % nx] != 0
            if live:
                (near if touches else plain).append(q - (1 << 31) if touches else q)
        return near + plain

    eight = tiles(8)
    if precision == 0 and len(eight) <= 3 * sm:
        return [8] + eight
    return [4] + tiles(4)


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    from paper_0812_1282_gb300 import _build

    lib = _build.build()
    tmp = tmp_path_factory.mktemp("tiles")
    (tmp / "main.cu").write_text(MAIN)
    out = str(tmp / "tiles")
    subprocess.run([_build.nvcc(), "-std=c++17", "-I", CSRC, str(tmp / "main.cu"), lib, "-o", out,
                    "-Xlinker", "-rpath=" + os.path.dirname(lib)], check=True, timeout=300)
    return out


def maps():
    rng = np.random.default_rng(5)
    for nx, ny in [(3, 3), (31, 4), (32, 8), (33, 9), (64, 5), (70, 30), (97, 17)]:
        for fill in (0.0, 0.004, 0.05, 0.97, 1.0):
            cls = (rng.random((ny, nx)) < fill).astype(np.uint8) * rng.integers(1, 8, (ny, nx), np.uint8)
            yield cls
        wall = np.zeros((ny, nx), np.uint8)
        wall[0] = wall[-1] = KNODEWALL
        yield wall
        edge = np.zeros((ny, nx), np.uint8)
        edge[-1, -1] = 2  # seen across both periodic edges
        yield edge


def test_tile_lists(exe):
    cases = [(precision, sm, cls, walls) for cls in maps() for walls in (0, 1)
             for precision, sm in ((0, 152), (0, 1), (1, 152))]
    text = "".join("%d %d %d %d %d\n%s\n" % (p, sm, c.shape[1], c.shape[0], w,
                                             " ".join(map(str, c.ravel())))
                   for p, sm, c, w in cases)
    out = subprocess.run([exe], input=text, check=True, capture_output=True, text=True,
                         timeout=300).stdout.splitlines()
    assert len(out) == len(cases)
    for line, (p, sm, c, w) in zip(out, cases):
        assert [int(v) for v in line.split()] == expected(p, sm, c, w)

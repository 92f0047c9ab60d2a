"""The launchers of the small-lattice steps refuse the shapes their kernels are
not made for, before anything is launched.  Host only: a shape that is not
refused ends at the missing device here, so this is not run beside one."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0812_1282_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include "lb_small.h"
int main()
{
    for (int storage = 0; storage < 3; ++storage)  // FP64, FP32, FP32 with compact g
        for (int rows = 0; rows <= 9; ++rows) {
            lbfe::DomDesc d{};
            d.nx = d.ny = 64;
            d.pitch = 96;
            d.compact = storage == 2;
            std::printf("step %d %d %d\n", storage, rows,
                        lbfe::launch_small_step(storage == 0, 1, d, nullptr, nullptr, 0, 0, rows, nullptr));
        }
    for (int steps = 1; steps <= 9; ++steps)
        for (int rows : {0, 1, 8, 9, 20, 21})
            for (int n : {3, 4, 5, 6, 7, 8, 64})
                for (int wide = 0; wide < 2; ++wide) {
                    lbfe::DomDesc d{};
                    d.nx = wide ? 64 : n;
                    d.ny = wide ? n : 64;
                    d.pitch = 96;
                    std::printf("steps %d %d %d %d\n", steps, rows, n,
                                lbfe::launch_small_steps(1, d, 0, steps, rows, nullptr));
                }
}
"""
INVALID = 1  # cudaErrorInvalidValue


@pytest.fixture(scope="module")
def codes(tmp_path_factory):
    import torch

    if torch.cuda.is_available():
        pytest.skip("a CUDA device is present")
    from paper_0812_1282_gb300 import _build

    lib = _build.build()
    tmp = tmp_path_factory.mktemp("ranges")
    (tmp / "main.cu").write_text(MAIN)
    exe = str(tmp / "ranges")
    subprocess.run([_build.nvcc(), "-std=c++17", "-I", CSRC, str(tmp / "main.cu"), lib, "-o", exe,
                    "-Xlinker", "-rpath=" + os.path.dirname(lib)], check=True, timeout=300)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    return [line.split() for line in out.splitlines()]


def test_one_step(codes):
    lowest = [1, 3, 1]  # FP32 full storage takes the halo in one round of its threads
    seen = 0
    for kind, *v in codes:
        if kind == "step":
            storage, rows, code = map(int, v)
            assert (code == INVALID) == (not lowest[storage] <= rows <= 8), v
            seen += 1
    assert seen == 30


def test_several_steps(codes):
    seen = 0
    for kind, *v in codes:
        if kind == "steps":
            steps, rows, n, code = map(int, v)
            fits = 2 <= steps <= 8 and rows >= 1 and 32 * (rows + 4 * (steps - 1)) <= 768
            assert (code == INVALID) == (not (fits and n >= 2 * steps)), v
            seen += 1
    assert seen == 9 * 6 * 7 * 2

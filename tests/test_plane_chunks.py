"""Planes per task of the FP32 3D pass (csrc/chunk3d.hpp), host code, against measurements: us a Faber
degree by planes per task on a GB300 (152 SMs, free surface), for sizes (nx, ny, nz) and damped
points.  The choice has to be no slower than chunks of 32 planes and within 10 % of the best chunk
measured (twice the model's rms error); and every chunk is between 1 and all planes."""
import os
import shutil
import subprocess

import pytest

MEASURED = {
    (192, 192, 192, 20): {192: 388, 96: 216, 64: 272, 48: 217, 39: 226, 32: 202, 28: 216, 24: 198, 22: 206, 20:
        195, 18: 196, 16: 191, 15: 196, 14: 189, 13: 195, 12: 191},
    (192, 192, 192, 40): {192: 398, 96: 227, 64: 296, 48: 227, 39: 234, 32: 215, 28: 219, 24: 214, 22: 208, 20:
        203, 18: 201, 16: 204, 15: 202, 14: 200, 13: 206, 12: 202},
    (64, 64, 64, 20): {64: 121, 32: 66, 22: 46, 16: 38, 13: 31},
    (100, 95, 260, 20): {260: 504, 130: 260, 87: 179, 65: 139, 52: 116, 44: 100, 38: 143, 33: 141, 29: 129, 26:
        120, 24: 109, 22: 103, 20: 132, 19: 122, 18: 119, 17: 112, 16: 107, 15: 101, 14: 95, 13: 120, 12: 109},
    (97, 113, 254, 20): {254: 495, 127: 255, 85: 176, 64: 137, 51: 116, 43: 180, 37: 157, 32: 141, 29: 129, 26:
        119, 24: 144, 22: 147, 20: 134, 19: 131, 17: 120, 16: 138, 15: 133, 14: 126, 13: 118, 12: 131},
    (130, 250, 90, 30): {90: 193, 45: 177, 30: 129, 23: 135, 18: 148, 15: 132, 13: 137, 12: 135},
    (128, 128, 128, 30): {128: 258, 64: 138, 43: 99, 32: 81, 26: 119, 22: 103, 19: 90, 16: 79, 15: 77, 13: 87,
        12: 86},
    (160, 160, 160, 30): {160: 324, 80: 173, 54: 204, 40: 160, 32: 130, 27: 162, 23: 142, 20: 159, 18: 145, 16:
        133, 15: 143, 14: 144, 13: 145, 12: 145},
    (251, 229, 197, 30): {197: 410, 99: 378, 66: 367, 50: 377, 40: 316, 33: 322, 29: 329, 25: 345, 22: 311, 20:
        317, 18: 328, 17: 334, 16: 330, 15: 318, 14: 323, 13: 330, 12: 322},
    (256, 256, 256, 30): {256: 536, 128: 488, 86: 473, 64: 461, 52: 457, 43: 470, 37: 419, 32: 424, 29: 430, 26:
        436, 24: 439, 22: 448, 20: 424, 19: 430, 18: 435, 16: 444, 15: 451, 14: 447, 13: 442, 12: 450},
    (227, 112, 249, 30): {249: 499, 125: 263, 83: 353, 63: 269, 50: 226, 42: 259, 36: 223, 32: 201, 28: 240, 25:
        217, 23: 243, 21: 229, 20: 223, 18: 229, 17: 224, 16: 211, 15: 217, 14: 215, 13: 209, 12: 214},
    (215, 141, 197, 30): {197: 398, 99: 216, 66: 284, 50: 218, 40: 244, 33: 225, 29: 224, 25: 222, 22: 218, 20:
        215, 18: 211, 17: 208, 16: 208, 15: 205, 14: 208, 13: 209, 12: 208},
    (256, 128, 128, 30): {128: 263, 64: 145, 43: 175, 32: 152, 26: 168, 22: 144, 19: 130, 16: 147, 15: 140, 13:
        142, 12: 136},
    (154, 188, 225, 30): {225: 449, 113: 240, 75: 321, 57: 242, 45: 267, 38: 246, 33: 246, 29: 238, 25: 239, 23:
        233, 21: 227, 19: 228, 18: 223, 17: 224, 15: 230, 14: 223, 13: 229, 12: 216},
    (400, 400, 400, 30): {400: 2120, 200: 1682, 134: 1531, 100: 1650, 80: 1562, 67: 1513, 58: 1567, 50: 1556,
        45: 1527, 40: 1551, 37: 1554, 34: 1543, 31: 1529, 29: 1558, 27: 1552, 25: 1543, 24: 1561, 23: 1576, 22:
        1572, 20: 1586, 19: 1596, 18: 1593, 17: 1602, 16: 1616, 15: 1629, 14: 1645, 13: 1662},
}

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "chunk3d.hpp"
int main(int argc, char** argv) {     // nx ny nz pml fs, any number of times: one problem each
    std::vector<ewv::Grid3> g;
    for (int a = 1; a + 4 < argc; a += 5)
        g.push_back({std::atoi(argv[a]), std::atoi(argv[a + 1]), std::atoi(argv[a + 2]), std::atoi(argv[a + 3]),
                     std::atoi(argv[a + 4]) != 0});
    std::printf("%d\n", ewv::planes_per_task(g, 152, 64, 8, 4));
}
"""


@pytest.fixture(scope="module")
def choose(repo_root, tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("chunk")
    src, exe = d / "c.cpp", d / "c"
    src.write_text(SOURCE)
    include = os.path.join(repo_root, "paper_2401_16322_gb300", "csrc")
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", include, str(src), "-o", str(exe)], check=True)

    def run(*grids):
        args = [str(int(v)) for g in grids for v in g]
        return int(subprocess.run([str(exe)] + args, capture_output=True, text=True, check=True).stdout)
    return run


@pytest.mark.parametrize("size", list(MEASURED))
def test_choice_is_near_the_best_measured(choose, size):
    us = MEASURED[size]
    kc = choose((*size, True))
    assert kc in us, kc
    assert us[kc] <= 1.10 * min(us.values()), (kc, us[kc], min(us.values()))
    former = [k for k in us if -(-size[2] // k) == -(-size[2] // 32)]     # as many chunks as of 32 planes
    assert us[kc] <= 1.01 * min(us[k] for k in former)


@pytest.mark.parametrize("grids", [[(12, 12, 12, 3, True)], [(2, 2, 2, 0, False)], [(64, 8, 7, 40, True)],
                                   [(400, 400, 400, 30, True)], [(192, 192, 192, 0, False)],
                                   [(64, 17, 15, 5, True), (200, 90, 300, 30, False), (9, 9, 2, 4, True)]])
def test_every_size_has_a_chunk(choose, grids):
    assert 1 <= choose(*grids) <= max(g[2] for g in grids)

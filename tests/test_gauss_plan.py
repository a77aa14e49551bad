"""The FP32 Gaussian stage's choice of tile and K splits (csrc/gauss_plan.cuh): the splits cover K, and at measured
shapes the choice is at most 10% slower than the fastest of the measured forms. Host code, compiled here."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2105_11004_gb300", "csrc")

# (m, d, s): {(wide, splits): us} on one GB300
MEASURED = {
    (32, 8, 512): {(0, 8): 15.6, (0, 4): 22.5, (0, 2): 36.7},
    (40, 20, 32768): {(0, 512): 67.1, (0, 256): 49.7, (0, 128): 45},
    (64, 20, 65536): {(0, 608): 93.5, (0, 512): 94.2, (0, 256): 76},
    (80, 20, 1600): {(0, 25): 17.4, (0, 13): 24, (0, 7): 36.1},
    (96, 48, 32768): {(0, 512): 68.5, (0, 256): 51.1, (0, 128): 47.1},
    (128, 64, 2048): {(0, 32): 18.6, (0, 16): 26, (0, 8): 40.5},
    (400, 100, 32768): {(0, 152): 120.2, (0, 128): 136.5, (1, 76): 163.6},
    (512, 128, 8192): {(0, 128): 51, (0, 64): 44.6, (0, 32): 45.1, (1, 76): 52.6, (1, 64): 55.2, (1, 32): 51.6},
    (528, 132, 2048): {(0, 32): 36.5, (0, 16): 42.4, (0, 8): 44.8, (1, 32): 34.1, (1, 16): 31.2, (1, 8): 51.3},
    (400, 200, 20000): {(0, 76): 134.6, (1, 76): 110.2},
    (800, 200, 20000): {(0, 44): 249.1, (1, 43): 198.9},
    (512, 256, 4096): {(0, 64): 48.8, (0, 32): 44.4, (0, 16): 44.6, (1, 64): 37.8, (1, 32): 34.2, (1, 16): 52.7},
    (1024, 256, 65536): {(0, 38): 793.4, (1, 38): 681},
    (600, 300, 8192): {(0, 41): 126.2, (0, 32): 130.2, (1, 30): 111},
    (1200, 300, 32768): {(0, 21): 851.6, (1, 15): 835.1},
    (768, 384, 4096): {(0, 34): 75.9, (0, 32): 74.2, (0, 16): 70.2, (1, 25): 73.3, (1, 16): 97.3},
    (2048, 512, 32768): {(0, 10): 1852.5, (1, 9): 1392.6},
    (1280, 640, 4096): {(0, 13): 192.2, (1, 10): 155.8},
    (1536, 768, 1600): {(0, 9): 114.4, (0, 7): 116.4, (1, 8): 84.4, (1, 7): 96},
    (3584, 896, 32768): {(0, 4): 5443.5, (1, 2): 6090.3},
    (2048, 1024, 2048): {(0, 5): 248.8, (1, 4): 194.4},
    (4096, 1024, 20000): {(0, 3): 4256.3, (1, 2): 3733.5},
}


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "p.cpp").write_text('#include <cstdio>\n#include "gauss_plan.cuh"\nint main() { long m, d, s;\n'
                             ' while (scanf("%ld %ld %ld", &m, &d, &s) == 3) {\n'
                             '  const lev::GaussPlan p = lev::gauss_plan(m, d, s);\n'
                             '  printf("%d %ld %ld\\n", (int)p.wide, (long)p.splits, (long)p.kchunk); } }\n')
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "p.cpp"), "-o", str(d / "p")], check=True)

    def run(shapes):
        text = "\n".join("%d %d %d" % t for t in shapes)
        out = subprocess.run([str(d / "p")], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(int(x) for x in line.split()) for line in out.splitlines()]
    return run


def test_splits_cover_k(plan):
    shapes = [(m, d, s) for d in list(range(4, 1025, 20)) + [1, 99, 129, 130, 257, 258, 516, 4096]
              for m in (1, d, 2 * d, 4 * d) for s in (1, 7, 256, 2048, 4098, 20011, 65536, 262144)]
    for (m, d, s), (wide, splits, kchunk) in zip(shapes, plan(shapes)):
        assert not wide or (d > 128 and d % 4 == 0 and s % 4 == 0), (m, d, s)
        assert splits >= 1 and splits * kchunk >= s and kchunk % (16 if wide else 8) == 0, (m, d, s)


def test_near_the_fastest_measured_form(plan):
    for shape, (wide, splits, _) in zip(MEASURED, plan(MEASURED)):
        us = MEASURED[shape]
        assert us[wide, splits] <= 1.1 * min(us.values()), shape

"""The FP32 Gaussian stage's choice of tile and K splits (csrc/gauss_plan.cuh): its time follows the rows of k
that the fullest SM goes through, so the 256-column tile is taken only where they are no more than the 128-column
tile's; and the splits cover K. Host code, compiled here."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2105_11004_gb300", "csrc")


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "p.cpp").write_text('#include <cstdio>\n#include "gauss_plan.cuh"\nint main() { long m, d, s;\n'
                             ' while (scanf("%ld %ld %ld", &m, &d, &s) == 3) {\n'
                             '  const lev::GaussPlan p = lev::gauss_plan(m, d, s), q = lev::gauss_plan_of(false, m, d, s);\n'
                             '  printf("%d %ld %ld %ld %ld\\n", (int)p.wide, (long)p.splits, (long)p.kchunk,'
                             ' (long)p.steps(), (long)q.steps()); } }\n')
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "p.cpp"), "-o", str(d / "p")], check=True)

    def run(shapes):
        text = "\n".join("%d %d %d" % t for t in shapes)
        out = subprocess.run([str(d / "p")], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(int(x) for x in line.split()) for line in out.splitlines()]
    return run


def test_no_more_work_than_the_narrow_tile(plan):
    shapes = [(m, d, s) for d in list(range(4, 1025, 20)) + [99, 129, 130, 256, 257, 258, 260, 384, 512, 516, 640, 1000]
              for m in (d, 2 * d, 3 * d + 1, 4 * d) for s in (256, 2048, 4096, 4098, 16384, 20011, 32768, 65536)]
    for (m, d, s), (wide, splits, kchunk, steps, narrow) in zip(shapes, plan(shapes)):
        assert not wide or (d > 128 and d % 4 == 0 and s % 4 == 0), (m, d, s)
        assert steps <= narrow, (m, d, s)
        assert splits * kchunk >= s and kchunk % (16 if wide else 8) == 0, (m, d, s)


def test_measured_shapes(plan):
    """Both sides measured: the wide tile is the faster one (or equal) at the first shapes, the slower at the others."""
    faster = [(1024, 256, 65536), (1024, 132, 65536), (1040, 260, 32768), (1536, 384, 32768), (2048, 512, 32768),
              (2560, 640, 32768), (4096, 1024, 32768), (520, 256, 4096), (264, 132, 2048)]
    slower = [(600, 300, 4096), (768, 384, 4096), (2064, 516, 32768), (3584, 896, 32768)]
    assert [p[0] for p in plan(faster + slower)] == [1] * len(faster) + [0] * len(slower)

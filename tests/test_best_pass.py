"""CPU check of the pass AUTO takes (csrc/rows_plan.h, best_pass): the lines it
draws, and bench.step_pass, which states the same rule for the bench's labels,
over extents, periods and storage formats."""
import itertools
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


@pytest.fixture(scope="module")
def best(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("best") / "best")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-I" + os.path.join(ROOT, "paper_1803_07822_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "best_pass_check.cpp"), "-o", exe])

    def run(cases):
        text = "".join("%d %d %d %d %d %d\n" % (*n, y, z, sb) for n, y, z, sb in cases)
        return subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split()
    return run


@pytest.mark.parametrize("n,zper,sb,want", [
    ((256, 256, 256), 0, 4, "fused"), ((256, 256, 96), 0, 4, "fused"), ((256, 256, 95), 0, 4, "rows"),
    ((256, 256, 32), 0, 4, "rows"), ((256, 256, 31), 0, 4, "flat"), ((128, 256, 128), 0, 4, "rows"),
    ((256, 256, 16), 1, 4, "rows"), ((256, 256, 15), 1, 4, "flat"), ((256, 256, 256), 1, 4, "rows"),
    ((256, 256, 96), 0, 2, "rows"), ((256, 256, 95), 0, 2, "flat"), ((256, 256, 32), 1, 2, "rows"),
    ((256, 256, 31), 1, 2, "flat"),
    ((252, 256, 256), 0, 4, "flat"), ((192, 256, 256), 0, 4, "flat"), ((64, 512, 512), 0, 4, "flat"),  # tiles not full, or of four rows
    ((128, 1, 60000), 1, 4, "flat"), ((260, 256, 256), 0, 4, "flat")])
def test_lines(best, n, zper, sb, want):
    assert best([(n, 1, zper, sb)]) == [want]


def test_the_bench_states_the_same_rule(best):
    import bench
    name = {4: "fp32", 2: "fp16"}
    cases = [((a, b, c), 1, z, sb) for a, b, c, z, sb in itertools.product(
        (4, 8, 64, 100, 128, 130, 192, 252, 256, 260), (1, 3, 64, 256), (3, 16, 64, 255, 256), (0, 1), (2, 4))]
    cases = [c for c in cases if c[0][0] * c[0][1] * c[0][2] >= 256]
    got = best(cases)
    want = [bench.step_pass(n, name[sb], "auto", bool(z)) for n, _, z, sb in cases]
    assert got == want

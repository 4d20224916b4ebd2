"""How a P2P work plan gets its scratch: whole pieces where the parts of small systems find no room."""
import os
import subprocess

import pytest

from paper_1405_2255_gb300 import build

CSRC = os.path.join(os.path.dirname(os.path.abspath(build.__file__)), "csrc")

HOST = r"""
#include <stdio.h>
#include <stdlib.h>
#include "plan_run.cuh"
// memory at hand, the most there is, the plan's fixed part, what it needs with parts and whole (-1: too large)
int main(int argc, char** argv) {
    size_t have = atoll(argv[1]), most = atoll(argv[2]), fixed = atoll(argv[3]), need[2] = {(size_t)atoll(argv[4]), (size_t)atoll(argv[5])};
    const bool parts = atoi(argv[6]);
    int ran = -1;
    const gb3::PlanEnd end = gb3::run_plan(
        fixed, parts,
        [&](bool p) {
            if (have < fixed) return fixed;
            const size_t n = need[p ? 0 : 1];
            if (n != ~(size_t)0 && n <= have) ran = p;
            return n;
        },
        [&](size_t b) {
            if (b <= have) return 0;
            have = b <= most ? b : 0;  // (a failing growth has given back what there was)
            return have ? 0 : -2;
        },
        [&] { return have; });
    printf("%d %d\n", (int)end, ran);
}
"""

RAN, TOO_LARGE, NO_ROOM = 0, 1, 2


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cu").write_text(HOST)
    subprocess.run([build.nvcc(), "-std=c++17", "-I", CSRC, "-o", str(d / "plan"), str(d / "plan.cu")], check=True,
                   capture_output=True)
    return str(d / "plan")


@pytest.mark.parametrize("have,most,parts,whole,share,end,ran", [
    (100, 100, 80, 50, 1, RAN, 1),         # at hand
    (0, 1000, 800, 500, 1, RAN, 1),        # after growing
    (0, 600, 800, 500, 1, RAN, 0),         # room for whole pieces only
    (0, 1000, -1, 500, 1, RAN, 0),         # too many records for parts
    (0, 1000, -1, -1, 1, TOO_LARGE, -1),
    (0, 100, 800, 500, 1, NO_ROOM, -1),
    (0, 5, 800, 500, 1, NO_ROOM, -1),      # not even the fixed part
    (0, 1000, 800, 500, 0, RAN, 0),        # no small system
])
def test_run_plan(exe, have, most, parts, whole, share, end, ran):
    out = subprocess.run([exe, *map(str, (have, most, 10, parts, whole, share))], capture_output=True, text=True)
    assert out.stdout.split() == [str(end), str(ran)]

"""Where lb_step_record may store states in place: the choice by precision, width and
address, on the host."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "lbm_internal.h"
int main(int, char** v) {
  lb_params p{};
  p.precision = std::atoi(v[1]), p.nx = std::atoi(v[2]), p.ny = std::atoi(v[3]);
  const size_t elem = p.precision == LB_FP64 ? 8 : p.precision == LB_FP32 ? 4 : 2;
  const bool tensor = std::atoi(v[4]) != 0;
  for (uintptr_t at = 4096; at < 4112; ++at)
    std::printf("%d%d ", lbm::record_in_place(p, at, 9 * elem * p.nx * p.ny, tensor), lbm::record_by_elements(p, at));
}
"""


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    d = tmp_path_factory.mktemp("record")
    (d / "r.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_1809_02390_gb300", "csrc"), str(d / "r.cpp"), "-o", str(d / "r")],
                   check=True)
    return lambda *a: [w for w in subprocess.run([str(d / "r"), *map(str, a)], check=True, capture_output=True,
                                                 text=True).stdout.split()]


# (precision, nx, ny, tensor copies): the alignment that stores in place need, that of single elements.
@pytest.mark.parametrize("case,place,element", [((2, 100, 80, 0), 4, 2), ((2, 101, 80, 0), 2, 2),
                                                ((1, 100, 80, 0), 4, 4), ((1, 101, 81, 0), 4, 4),
                                                ((0, 70, 33, 0), 8, 8), ((1, 1000, 700, 1), 16, 4),
                                                ((2, 1000, 704, 1), 16, 2)])
def test_alignment(choose, case, place, element):
    for at, w in enumerate(choose(*case)):
        assert w == f"{int(at % place == 0)}{int(at % element == 0)}", at

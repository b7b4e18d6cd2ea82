"""The device-resident CG's step rule (csrc/cg_rule.h) on the CPU: ordinary steps, curvatures at the rounding level
and non-finite ones, and what a first step does with them in a Newton system and in an adjoint solve; and that the
held-out gradient's solves ask for the latter."""
import os
import re

import pytest

import host_cpp

SOURCE = r"""
#include <cstdio>
#include "cg_rule.h"
int main() {
  double pAp, floor, rz;
  int first, unit;
  while (std::scanf("%lf %lf %lf %d %d", &pAp, &floor, &rz, &first, &unit) == 5) {
    const kqr::CgStep s = kqr::cg_step_rule(pAp, floor, rz, first != 0, unit != 0);
    std::printf("%.17g %d\n", s.a, s.state);
  }
}
"""
RUN, TRUNC, NONFINITE = 0, 2, 3
CASES = [  # pAp, floor, rz, first, unit_first -> step, state
    ((4.0, 0.0, 2.0, 1, 1), (0.5, RUN)), ((4.0, 3.9, 2.0, 0, 0), (0.5, RUN)),
    ((3.9, 3.9, 2.0, 1, 1), (1.0, TRUNC)), ((3.9, 3.9, 2.0, 0, 1), (0.0, TRUNC)),
    ((0.0, 0.0, 2.0, 1, 1), (1.0, TRUNC)), ((-1.0, 0.0, 2.0, 1, 1), (1.0, TRUNC)),
    ((0.0, 0.0, 2.0, 1, 0), (0.0, TRUNC)), ((-1.0, 0.0, 2.0, 1, 0), (0.0, TRUNC)), ((-1.0, 0.0, 2.0, 0, 0), (0.0, TRUNC)),
    (("nan", 0.0, 2.0, 1, 1), (0.0, NONFINITE)), (("inf", 0.0, 2.0, 0, 1), (0.0, NONFINITE)),
    (("-inf", 0.0, 2.0, 1, 0), (0.0, NONFINITE))]


def test_step_rule(tmp_path):
    out = host_cpp.run(SOURCE, tmp_path, "\n".join(" ".join(map(str, c)) for c, _ in CASES)).split("\n")
    for (case, (a, state)), line in zip(CASES, out):
        got = line.split()
        assert (float(got[0]), int(got[1])) == (a, state), case


def test_adjoint_solves_keep_x_at_a_non_positive_first_curvature():
    text = open(os.path.join(host_cpp.CSRC, "grad.cu")).read()
    adjoint = text[text.index("static kqr_status adjoint_cg("):]
    adjoint = adjoint[:adjoint.index("\n}\n")]
    assert re.search(r"\.unit_first = false;", adjoint)

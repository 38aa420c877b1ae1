"""Which stage-kernel form a handle takes, with launches that the device rejects (CPU).

csrc/stage_forms.h is compiled on its own, with given times in place of launches (negative: rejected).
"""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_02858_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "stage_forms.h"
// fp32 q status-of-form-1 us...: prints the status, the form and which forms were timed
int main(int argc, char** argv) {
  double us[10];
  for (double& x : us) x = -1;
  int form = 99, timed = 0;
  const int rc = cmcg::choose_form(std::atoi(argv[1]) != 0, std::atoi(argv[2]), us, &form, [&](int f, double* t) {
    timed |= 1 << f;
    *t = std::atof(argv[4 + f]);
    return f == 1 ? std::atoi(argv[3]) : 0;
  });
  std::printf("%d %d %d\n", rc, form, timed);
}
"""


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    d = tmp_path_factory.mktemp("forms")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(d / "t.cpp"), "-o", str(d / "t")], check=True)

    def run(fp32, q, us, status=0):
        us = [*us, *[-1] * (10 - len(us))]
        out = subprocess.run([str(d / "t"), *map(str, (int(fp32), q, status, *us))], check=True, capture_output=True,
                             text=True).stdout.split()
        return int(out[0]), int(out[1]), [f for f in range(10) if int(out[2]) >> f & 1]

    return run


@pytest.mark.parametrize("fp32,q,us,form,timed", [
    (True, 1, [3, 2, 4, 5, 6, 7, 1], 1, range(6)),          # the tensor-core form is not a candidate
    (True, 2, [3, 3, 4, 5, -1, 2.5, 1], 5, range(6)),
    (True, 2, [3, 3, 4, 5, 6, 7, 1], 0, range(6)),          # ties: the first
    (True, 3, [3, 2, 4, 5, 6, 7, 90], 6, [6]),              # P3: that form whatever it takes
    (True, 3, [3, 2, 4, 5, 6, 7, -1], 1, range(7)),         # rejected: one of the others
    (True, 3, [-1, -1, 4, -1, 6, 7, -1], 2, range(7)),
    (True, 3, [-1] * 7, -1, range(7)),                      # nothing can be launched
    (True, 1, [-1] * 6 + [1], -1, range(6)),
    (False, 1, [3, 2, 4, 1], 1, range(3)),
    (False, 3, [-1, -1, 4], 2, range(3)),
    (False, 3, [-1, -1, -1], -1, range(3)),
])
def test_choice(choose, fp32, q, us, form, timed):
    assert choose(fp32, q, us) == (0, form, list(timed))


def test_a_failure_is_passed_on(choose):
    rc, _, timed = choose(True, 1, [3, 2, 4, 5, 6, 7], status=-8)
    assert rc == -8 and timed == [0, 1]

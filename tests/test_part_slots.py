"""The slots through which a block of the resident solvers hands over its sums
(csrc/ulp_parts.h), on the host.  Between the barriers of a phase any two sums of a block can
follow each other with nothing between them (one map has stopped, another is in a phase with a
single sum), so no two may share a slot."""
import os
import subprocess

import paper_2203_13675_gb300

CSRC = os.path.join(os.path.dirname(paper_2203_13675_gb300.__file__), "csrc")

PROGRAM = r"""
#include <cstdio>
#include "ulp_parts.h"

int main() {
  bool taken[ulp::kPartSlots] = {};
  for (int place = 0; place < ulp::kResMaxWarps; ++place)
    for (int sum = 0; sum < 3; ++sum) {
      const int s = ulp::part_slot(place, sum);
      if (s < 0 || s >= ulp::kPartSlots || taken[s]) {
        std::printf("place %d, sum %d: slot %d\n", place, sum, s);
        return 1;
      }
      taken[s] = true;
    }
}
"""


def test_every_sum_of_a_block_has_its_own_slot(tmp_path):
    src, exe = tmp_path / "slots.cpp", tmp_path / "slots"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

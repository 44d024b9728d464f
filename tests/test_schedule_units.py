"""The tile planners with more persistent units than a schedule table can name (a part with more SMs): no table, round-robin,
and nothing written past the planners' fixed arrays.  The header is host code, compiled and run here with the address sanitizer."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_04732_b200", "csrc")

PROGRAM = r"""
#include "schedule.cuh"
#include <cstdlib>
#include <cstdio>
using namespace flop::tc;
int main(int argc, char** argv) {
  const int units = atoi(argv[1]);
  std::vector<ItemGroup> groups;      // uneven costs, more items than units
  groups.push_back(ItemGroup{48.0, 0, 0, 0, 2 * units + 1, 1});
  groups.push_back(ItemGroup{12.0, 0, 1, 2 * units + 1, units, 1});
  double rr = -1.0;
  const bool keep = round_robin_is_good(groups, units, &rr);
  static Schedule s;
  s.n_units = 7;
  const double makespan = keep ? 0.0 : deal_groups(groups, 3 * units + 1, units, kSchedProblemShift, &s);
  printf("%d %d %d\n", (int)keep, (int)(makespan > 0.0 && makespan <= rr), keep ? 0 : s.n_units);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("schedule")
    (d / "main.cpp").write_text(PROGRAM)
    exe = str(d / "main")
    subprocess.run(["g++", "-std=c++17", "-O1", "-g", "-fsanitize=address", "-I" + CSRC, "-o", exe, str(d / "main.cpp")], check=True)
    return exe


@pytest.mark.parametrize("units", [1, 74, 148, 149, 152, 1000])
def test_units_beyond_the_table(program, units):
    r = subprocess.run([program, str(units)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    keep, balanced, n = (int(v) for v in r.stdout.split())
    if units > 148:
        assert keep == 1
    elif not keep:
        assert balanced == 1 and n == units

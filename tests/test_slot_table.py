"""The table of the device's answers behind the on-chip plans (host C++, CPU
only): a failed query is asked again, a shape that does not fit is not, and
the table stays bounded.  Every table of such answers in the sources is this one."""
import os
import re
import shutil
import subprocess

import pytest

from tests.test_kernel_sources import CSRC, SOURCES

PROGRAM = r"""
#include <cstdio>
#include <tuple>
#include "slot_table.h"
int main() {
  cbdg::SlotTable<std::tuple<int, int>> t;
  int asked = 0;
  auto answer = [&](int n) { return [&asked, n] { ++asked; return n; }; };
  if (t.get({0, 1}, answer(-1)) != -1 || t.get({0, 1}, answer(7)) != 7 || asked != 2) return 1;  // not kept
  if (t.get({0, 1}, answer(9)) != 7 || asked != 2) return 2;                                     // kept
  if (t.get({1, 1}, answer(0)) != 0 || t.get({1, 1}, answer(3)) != 0 || asked != 3) return 3;    // kept
  for (int k = 0; k < 100000; ++k) t.get({2, k}, answer(5));
  return t.size() <= 4096 ? 0 : 4;
}
"""


@pytest.mark.skipif(not shutil.which("g++"), reason="needs g++")
def test_failures_are_asked_again_and_the_table_is_bounded(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-I" + CSRC, str(src), "-o", exe, "-pthread"], check=True)
    assert subprocess.run([exe]).returncode == 0


def test_occupancy_answers_are_kept_in_that_table():
    for path in SOURCES:
        text = open(path).read()
        assert not re.search(r"static std::map", text), os.path.basename(path)
        # a query that failed is told apart from a shape that does not fit
        for m in re.finditer(r"cudaOccupancyMaxActiveClusters\(.*?return n;", text, re.S):
            assert "return -1;" in m.group(0), os.path.basename(path)

"""The launch form of the lean mixed column depends on the levels as well as the columns: a tile's
shared memory decides how many of them an SM holds."""
import os
import shutil
import subprocess

import pytest

from tests.conftest import ROOT

TILE4, TILE8, COLUMN1, COLUMN2 = 6, 8, 10, 12
# (bisections, levels, terrain): the fastest form measured on a GB300, or within 4 per cent of it
FASTEST = {(2, 256, 0): TILE8, (3, 20, 0): TILE8, (3, 180, 0): TILE8, (3, 180, 1): TILE8, (3, 256, 1): TILE8,
           (4, 20, 0): TILE4, (4, 60, 0): TILE4, (4, 69, 0): TILE4, (4, 70, 0): TILE8, (4, 88, 0): TILE8,
           (4, 128, 0): TILE8, (4, 174, 0): TILE8, (4, 180, 0): COLUMN2, (4, 256, 0): COLUMN2,
           (4, 20, 1): TILE4, (4, 57, 1): TILE4, (4, 58, 1): COLUMN1, (4, 128, 1): COLUMN1, (4, 180, 1): COLUMN1,
           (4, 256, 1): COLUMN1, (5, 60, 0): COLUMN2, (5, 256, 0): COLUMN2, (5, 60, 1): COLUMN1, (7, 90, 0): COLUMN2}
SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "lean_rule.h"
int main(int argc, char** argv) {
  for (int i = 1; i + 2 < argc; i += 3)
    printf("%d\n", icon::lean_form_for(20ll << (2 * atoi(argv[i]) + 2), atoi(argv[i + 1]), atoi(argv[i + 2]), 152,
                                       233472, 1024));
  return 0;
}
"""


def test_form_follows_columns_and_levels(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_2511_02021_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    out = subprocess.run([str(exe)] + [str(v) for k in FASTEST for v in k], check=True, capture_output=True,
                         text=True).stdout.split()
    assert dict(zip(FASTEST, map(int, out))) == FASTEST

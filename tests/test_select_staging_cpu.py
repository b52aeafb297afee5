"""The selection kernel's staging buffer: every 16-byte group that a pass reads lies inside the words the launch asks for."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_12335_b200", "csrc")

PROGRAM = r"""
#include "select_staging.h"
#include <cstdio>
int main() {
  for (int n = 1; n <= 41000; n += n < 300 ? 1 : 97)
    for (int pad = 0; pad < 4; ++pad)
      if (4 * vatp::staged_groups(pad, n) > vatp::staged_words(n) || pad + n > 4 * vatp::staged_groups(pad, n)) {
        std::printf("n %d pad %d: groups end at word %d of %d\n", n, pad, 4 * vatp::staged_groups(pad, n), vatp::staged_words(n));
        return 1;
      }
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a C++ compiler")
def test_every_group_read_is_inside_the_buffer(tmp_path):
    src, exe = tmp_path / "staging.cpp", tmp_path / "staging"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

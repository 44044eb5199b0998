"""The tags of whole calls in the status words: 48 bits, never repeated (the numbers of calls
that a 64-bit mix cut to 48 bits got through without a repeat were a few million)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_18954_gb300", "csrc")

PROGRAM = r"""
#include <algorithm>
#include <cstdio>
#include <vector>
#include "gpo_tag.cuh"
int main() {
  const uint64_t starts[] = {0, (1ull << 32) - 4000000, (1ull << 47) - 4000000};
  std::vector<uint64_t> t;
  for (uint64_t s : starts)
    for (uint64_t n = s; n < s + 8000000; ++n) t.push_back(gpo::tag_of(n));
  std::sort(t.begin(), t.end());
  const bool unique = std::adjacent_find(t.begin(), t.end()) == t.end();
  std::printf("%d %d\n", (int)unique, (int)(t.back() >> 48 == 0));
}
"""


def test_tags_do_not_repeat(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    src = tmp_path / "tags.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "tags"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)])
    assert subprocess.check_output([str(exe)], text=True).split() == ["1", "1"]

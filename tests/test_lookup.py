"""A number looked up at first use (the CTA pairs that a device holds): kept once found, asked for
again after a lookup that failed.  CPU, with a fake lookup."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include "sp_lookup.h"
int main() {
  std::atomic<int> kept{0};
  int calls = 0, answer = 0;
  auto lookup = [&] { ++calls; return answer; };
  if (sp::kept_or_looked_up(kept, lookup) != 0 || calls != 1) return 1;
  answer = -1;
  if (sp::kept_or_looked_up(kept, lookup) != 0 || calls != 2) return 2;  // failed before: asked again
  answer = 76;
  if (sp::kept_or_looked_up(kept, lookup) != 76 || calls != 3) return 3;
  answer = 0;
  if (sp::kept_or_looked_up(kept, lookup) != 76 || calls != 3) return 4;  // kept
  return 0;
}
"""


def test_a_failed_lookup_is_not_kept(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "lookup.cpp", tmp_path / "lookup"
    src.write_text(HARNESS)
    subprocess.check_call([cxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_2405_03594_gb300", "csrc"), str(src), "-o",
                           str(exe)])
    assert subprocess.run([str(exe)]).returncode == 0


def test_the_pairs_are_looked_up_that_way():
    with open(os.path.join(ROOT, "paper_2405_03594_gb300", "csrc", "sp_linear_dense.cu")) as f:
        s = f.read()
    body = s[s.index("int resident_pairs(int dev)"):s.index("size_t round256(")]
    assert "kept_or_looked_up(" in body and ".store(" not in body

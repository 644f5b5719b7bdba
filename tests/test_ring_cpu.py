"""The operand ring's record of its last uses (csrc/ring.h), which a product kernel whose wait gave up needs to await the
copies in flight: compiled here and compared with a ring that is filled copy by copy."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = r'''
#include "ring.h"
#include <cstdio>
int main() {
  for (int stages = 1; stages <= 10; ++stages) {
    unsigned slot = 0, ph = 0;
    bool first = true;
    for (int issued = 0; issued <= 5 * stages; ++issued) {
      for (int s = 0; s < stages; ++s) std::printf("%d %d %d %d\n", stages, issued, s, xl::ring_last_use(slot, ph, first, s));
      if ((int)++slot == stages) {
        slot = 0;
        ph ^= 1;
        first = false;
      }
    }
  }
}
'''


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_last_use_of_every_slot(tmp_path):
    src = tmp_path / "ring.cpp"
    src.write_text(CODE)
    exe = tmp_path / "ring"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I" + os.path.join(ROOT, "paper_1705_10845_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    for line in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines():
        stages, issued, s, got = map(int, line.split())
        uses = [i // stages for i in range(issued) if i % stages == s]   # the phase that each use of slot s completes
        assert got == (uses[-1] & 1 if uses else -1), (stages, issued, s)

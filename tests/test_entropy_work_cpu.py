"""The sizing of the entropy's work area (csrc/entropy_work.h), compiled here with an allocator of a given size:
one area for all sizes, halved where it does not fit, none at all where one matrix does not."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = r'''
#include "entropy_work.h"
#include <cstdio>
#include <cstdlib>
using xl::EntropyWork;
static size_t room, held;
static int live;
struct Block { size_t n; };
static void* take(size_t n) {
  if (held + n > room) return nullptr;
  held += n;
  ++live;
  Block* b = static_cast<Block*>(std::malloc(sizeof(Block)));   // addresses only: nothing is stored through them
  b->n = n;
  return b;
}
static void give(void* p) {
  held -= static_cast<Block*>(p)->n;
  --live;
  std::free(p);
}
int main() {
  for (int np : {128, 512, 1024, 16384})
    for (int num = 0; num <= 24; ++num) {   // room for num / 2 matrices
      const size_t one = EntropyWork::per(np) * sizeof(double);
      room = one * num / 2;
      EntropyWork w;
      w.reserve(np, 11, take, give);
      const int most = (int)(((size_t)2 << 30) / one), full = most < 1 ? 1 : most < 11 ? most : 11;
      const double* end = w.cap ? w.part + (size_t)(np / 64) * w.cap : nullptr;
      const long used = w.cap ? (long)(end - w.mats) : 0;
      room = (size_t)1 << 40;
      EntropyWork v = w;   // the memory is back: the whole area
      v.reserve(np, 11, take, give);
      const int after = v.cap, blocks = live;
      v.reserve(128, 3, take, give);   // a smaller system uses what is there
      const int small = v.cap, blocks2 = live;
      v.free_all(give);
      std::printf("%d %d %d %d %ld %zu %d %d %d %d %d\n", np, num, full, w.cap, used, EntropyWork::per(np), after, blocks, small, blocks2, live);
    }
  static double a[128 * 128], b[128 * 128];
  const EntropyWork w = EntropyWork::on(a, b, 128);
  std::printf("%d %ld\n", w.cap, (long)(w.part + 2 - b));
}
'''


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_area_follows_the_memory(tmp_path):
    src = tmp_path / "area.cpp"
    src.write_text(CODE)
    exe = tmp_path / "area"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I" + os.path.join(ROOT, "paper_1705_10845_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    rows = [list(map(int, l.split())) for l in subprocess.run([str(exe)], capture_output=True, text=True, check=True)
            .stdout.splitlines()]
    cap, inside = rows.pop()
    assert cap == 1 and inside <= 128 * 128          # the engine's own matrices hold one
    assert len(rows) == 4 * 25
    for np_, num, full, cap, used, per, after, blocks, small, blocks2, live in rows:
        want = full                                  # halved until it fits
        while want > num // 2:
            want //= 2
        assert cap == want
        assert used == cap * per                     # the parts fill the area and no more
        assert after == full and blocks == 1
        assert small == 3 and blocks2 == 1
        assert live == 0

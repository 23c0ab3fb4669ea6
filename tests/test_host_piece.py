"""A host array is read in place only where one page-locked piece of memory holds all of it (checked without a GPU)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "host_piece.h"
#include <cassert>
#include <cstdint>
// page-locked pieces: bytes 1000-4999 and 9000-12999 of the address space, which the device sees 1 << 20 higher
static bool piece_of(const void* p, sjd::HostPiece* out) {
  const uintptr_t at = reinterpret_cast<uintptr_t>(p), pieces[2][2] = {{1000, 4000}, {9000, 4000}};
  for (auto& x : pieces)
    if (at >= x[0] && at < x[0] + x[1]) {
      out->device = reinterpret_cast<char*>(at + (1 << 20));
      out->start = reinterpret_cast<char*>(x[0] + (1 << 20));
      out->size = x[1];
      return true;
    }
  return false;
}
static uintptr_t ask(uintptr_t p, size_t n) {
  return reinterpret_cast<uintptr_t>(sjd::device_address_of(reinterpret_cast<void*>(p), n, piece_of));
}
int main() {
  assert(ask(1000, 4000) == 1000 + (1 << 20) && ask(1200, 3800) == 1200 + (1 << 20) && ask(12999, 1) == 12999 + (1 << 20));
  assert(ask(1000, 4001) == 0 && ask(4999, 2) == 0);   // runs past its piece
  assert(ask(1000, 12000) == 0 && ask(4000, 6000) == 0);  // both ends in a piece, a gap between them
  assert(ask(6000, 10) == 0 && ask(8990, 20) == 0);
  return 0;
}
"""


def test_only_one_piece_counts(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2512_07503_b200", "csrc"), str(src), "-o", str(exe)])
    subprocess.check_call([str(exe)])

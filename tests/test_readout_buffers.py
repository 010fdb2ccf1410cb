"""The buffers of a read-out after an allocation or an upload that failed: the next
call must find either nothing or a complete set (a pointer to an unfilled table of
offsets would be read on the device).  Compiled for the host, without CUDA."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_01047_gb300", "csrc")

CODE = r"""
#include <cassert>
#include <cstdint>
#include <cstdlib>
#include "readout.h"
int main() {
  for (int fail_alloc = 0; fail_alloc < 2; ++fail_alloc)
    for (int fail_fill = 0; fail_fill < 3; ++fail_fill) {
      dca::ReadoutBuffers b;
      double *out = nullptr, *tab = nullptr;
      long long* offsets = nullptr;
      int allocs = 0, fills = 0, calls = 0, rc = -1;
      while (rc != 0) {
        assert(++calls < 8);
        rc = b.prepare({{(void**)&out, 1000}, {(void**)&offsets, 24}, {(void**)&tab, 0}}, -3,
                       [&](size_t n) -> void* {
                         assert(n == 1024 + 256);
                         return allocs++ < fail_alloc ? nullptr : std::malloc(n);
                       },
                       [&]() -> int {
                         assert(out && offsets);
                         return fills++ < fail_fill ? -2 : 0;
                       });
        assert(b.ready == (rc == 0));
        if (rc == -3) assert(!out && !offsets);
      }
      assert(calls == 1 + fail_alloc + fail_fill && allocs == 1 + fail_alloc && fills == 1 + fail_fill);
      assert((char*)offsets == (char*)out + 1024);
      assert(b.prepare({}, -3, [](size_t) -> void* { std::abort(); }, []() -> int { std::abort(); }) == 0);
      std::free(b.base);
    }
  return 0;
}
"""


def test_a_failed_call_leaves_no_half_made_set(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(CODE)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    subprocess.run([str(exe)], check=True)


def test_the_read_outs_make_their_buffers_through_it():
    with open(os.path.join(CSRC, "walker.cu")) as f:
        text = f.read()
    for name in ("d_Gout", "d_Gbase", "d_Mout", "d_Mbase", "d_Mtab"):
        assert "%s = (" % name not in text  # no pointer set on its own

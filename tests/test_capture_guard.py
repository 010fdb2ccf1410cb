"""Capture of the window loop that stops on the way: no stream may be left
capturing (every later sweep of the handle would fail with a capture error and not
with the cause).  The guard is compiled for the host, without CUDA."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_01047_gb300", "csrc")

CODE = r"""
#include <cassert>
#include "capture_guard.h"
static int capturing[2], ended;
static int part(int stream, int fail_at, int step) {
  dca::CaptureGuard cap([&] { if (fail_at == step) return 7; ++capturing[stream]; return 0; },
                        [&] { --capturing[stream]; ++ended; return fail_at == step + 2 ? 9 : 0; });
  int e = cap.start();
  if (e != 0) return e;
  if (fail_at == step + 1) return 8;
  if (stream == 0) {
    e = part(1, fail_at, 10);  // the body of a node of this capture
    if (e != 0) return e;
  }
  return cap.finish();
}
int main() {
  const int steps[] = {-1, 0, 1, 2, 10, 11, 12};
  for (int f : steps) {
    ended = 0;
    const int e = part(0, f, 0);
    assert(capturing[0] == 0 && capturing[1] == 0);
    assert(e == (f < 0 ? 0 : f % 10 + 7));  // the cause, whatever the clean-up returned
    assert(ended == (f == 0 ? 0 : (f == 1 || f == 10 ? 1 : 2)));
  }
  return 0;
}
"""


def test_no_way_out_leaves_a_stream_capturing(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(CODE)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    subprocess.run([str(exe)], check=True)


def test_every_capture_of_the_window_loop_is_guarded():
    with open(os.path.join(CSRC, "walker.cu")) as f:
        text = f.read()
    for call in ("cudaStreamBeginCaptureToGraph(", "cudaStreamEndCapture("):
        assert text.count(call) == 1
    assert len(re.findall(r"auto cap = guard_capture\(h->cap", text)) == 2

"""Downloads of a device call's results (csrc/lorads_fetch.h) with a fake copy, compiled for the host:
a set error word, a failing copy and a failing wait each return their status and leave the caller's
buffers as they were; a good call fills the wanted ones."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2403_09133_gb300", "csrc")

PROGRAM = r"""
#include <cstring>
#include "lorads_fetch.h"
int main() {
  const double src[2] = {3.0, 4.0};
  // copies run only in wait(), as on a stream: the word must be waited for before it is read
  for (int mode = 0; mode < 4; ++mode) {     // good, error word set, failing copy, failing wait
    const int word = mode == 1;
    double u = -1.0, y = -1.0;
    struct { void* d; const void* s; size_t n; } queue[4];
    int queued = 0;
    auto copy = [&](void* d, const void* s, size_t n) {
      if (mode == 2) return -7;
      queue[queued++] = {d, s, n};
      return 0;
    };
    auto wait = [&] {
      if (mode == 3) return -8;
      for (int i = 0; i < queued; ++i) memcpy(queue[i].d, queue[i].s, queue[i].n);
      queued = 0;
      return 0;
    };
    const lorads::FetchItem items[3] = {{&u, src, 8}, {nullptr, src, 8}, {&y, src + 1, 8}};
    const int st = lorads::fetch_outputs(&word, items, 3, -5, copy, wait);
    const int want[4] = {0, -5, -7, -8};
    if (st != want[mode]) return 1;
    if (mode == 0 ? (u != 3.0 || y != 4.0) : (u != -1.0 || y != -1.0)) return 2;
  }
  return 0;
}
"""


def test_fetch_leaves_buffers_of_a_failed_call(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = tmp_path / "fetch.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "fetch"
    subprocess.run([cxx, "-O1", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o",
                    str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_forward_pass_fetches_behind_its_error_word():
    """The learned start's forward pass takes its outputs through fetch_outputs alone."""
    text = open(os.path.join(CSRC, "lorads_gnn.cu")).read()
    body = text[text.index("int lorads_gnn_forward("):text.index("int lorads_gnn_train_step(")]
    assert "fetch_outputs(" in body and body.count("cudaMemcpyAsync(") == 1

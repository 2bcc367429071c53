"""A step's first use under CUDA graphs (csrc/first_use.h), with CUDA calls that fail
on demand: once the step's launches are enqueued, its status is theirs, whatever
becomes of the capture; a capture that began is ended, its graph destroyed and the
error of the call that failed forgotten."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "first_use.h"
struct Fake {
  using Graph = int*;
  using Exec = int*;
  const char* fails;
  bool capturing = false, cleared = false;
  int graphs = 0, cell = 0;
  bool is(const char* what) const { return std::strcmp(fails, what) == 0; }
  bool begin() { return is("begin") ? false : (capturing = true); }
  bool end(Graph* g) {
    capturing = false;
    *g = is("end") ? nullptr : &cell;
    graphs += *g != nullptr;
    return !is("end") && !is("invalid");
  }
  bool instantiate(Exec* x, Graph g) {
    *x = g;
    return !is("instantiate");
  }
  void destroy(Graph) { --graphs; }
  void clear_error() { cleared = true; }
};
int main(int, char** argv) {
  Fake cu{argv[1]};
  int enqueued = 0, recorded = 0;
  int* exec = &enqueued;
  const int st = memspec::run_then_capture(cu, [&] {
    if (cu.capturing) return cu.is("record") ? 7 : (++recorded, 0);
    return cu.is("run") ? 5 : (++enqueued, 0);
  }, &exec);
  std::printf("%d %d %d %d %d %d", st, enqueued, exec != nullptr, cu.capturing, cu.graphs, cu.cleared);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("first_use")
    (d / "t.cpp").write_text(PROGRAM)
    csrc = os.path.join(ROOT, "paper_2608_10362_gb300", "csrc")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", csrc, str(d / "t.cpp"), "-o", str(d / "t")], check=True)
    return str(d / "t")


@pytest.mark.parametrize("fails,status,enqueued,captured,cleared", [
    ("nothing", 0, 1, 1, 0),
    ("run", 5, 0, 0, 0),             # the step itself: nothing is captured
    ("begin", 0, 1, 0, 1), ("record", 0, 1, 0, 1), ("end", 0, 1, 0, 1), ("invalid", 0, 1, 0, 1),
    ("instantiate", 0, 1, 0, 1),
])
def test_status_is_the_steps_own(program, fails, status, enqueued, captured, cleared):
    out = subprocess.run([program, fails], capture_output=True, text=True, check=True).stdout
    assert out.split() == [str(v) for v in (status, enqueued, captured, 0, 0, cleared)]

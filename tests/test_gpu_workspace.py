"""Workspace buffers that need not fit (the FP64 digit images): a request that
cannot be met drops the old buffer, so captured graphs that hold its address must
read as stale (the generation moves), and nothing is allocated while a graph is
captured.  Checked in a small program linked with the library."""
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SRC = r"""
#include <stdio.h>
#include "internal.h"
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
  const size_t huge = (size_t)1 << 50;  // more than any device has: the allocation fails
  cola::Ctx c;
  void* p = c.optional_ws("a", 4096);
  CHECK(p && c.ws.bufs.count("a"));
  const uint64_t g = c.ws.generation;
  CHECK(c.optional_ws("a", 1000) == p && c.ws.generation == g);
  c.capturing = true;
  CHECK(c.optional_ws("a", 4096) == p);
  CHECK(!c.optional_ws("a", 8192) && !c.optional_ws("b", 8));
  CHECK(c.ws.generation == g && c.ws.bufs.at("a").p == p && !c.ws.bufs.count("b"));
  c.capturing = false;
  CHECK(!c.ws.try_get("a", huge));
  CHECK(!c.ws.bufs.count("a") && c.ws.generation > g);
  CHECK(c.optional_ws("a", 4096));
  c.ws.release_all();
  return 0;
}
"""


def test_optional_buffers(tmp_path):
    from paper_2309_03060_gb300 import build
    lib = build.build()
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(SRC)
    r = subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-I", build.CSRC, str(src), lib,
                        "-Xlinker", f"-rpath={os.path.dirname(lib)}", "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr

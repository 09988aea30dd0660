"""The pool of optional device fields (image_pool.h) against an allocator with a limit: its bounds,
an allocation that fails part-way although there seemed to be room, no second attempt at a size
once asked for, and growth for a larger one."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "image_pool.h"
using pfmp::ImagePool;
static size_t limit, used, calls, mems;
static size_t free_bytes, total_bytes;
static void* take(size_t n) { ++calls; if (used + n > limit) return nullptr; used += n; return malloc(1); }
static size_t field;
static void give(void* p) { used -= field; free(p); }
static void mem(size_t* f, size_t* t) { ++mems; *f = free_bytes; *t = total_bytes; }
static int ask(ImagePool& P, int n) { return P.reserve(n, field, mem, take, give); }
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
int main() {
  field = 10;
  {  // everything fits: kept whole, then no call at all
    ImagePool P;
    free_bytes = 100000; total_bytes = 1000000; limit = 1000000; used = calls = mems = 0;
    CHECK(ask(P, 8) == 8 && used == 240 && calls == 24 && mems == 1);
    CHECK(ask(P, 8) == 8 && ask(P, 3) == 3 && calls == 24 && mems == 1);
    CHECK(ask(P, 10) == 10 && used == 300 && mems == 2);
  }
  {  // a quarter of the free memory
    ImagePool P;
    free_bytes = 1000; total_bytes = 1000000; limit = 1000000; used = 0;
    CHECK(ask(P, 64) == 8 && used == 240);
  }
  {  // a sixteenth of the device, what is held included
    ImagePool P;
    free_bytes = 1000000; total_bytes = 1600; limit = 1000000; used = 0;
    CHECK(ask(P, 2) == 2 && ask(P, 64) == 3 && used == 90);
  }
  {  // the allocation fails in the middle of an entry: given back, the same answer ever after
    ImagePool P;
    free_bytes = 100000; total_bytes = 1000000; limit = 145; used = calls = 0;
    CHECK(ask(P, 8) == 4 && used == 120);
    const size_t c = calls;
    limit = 1000000;
    CHECK(ask(P, 8) == 4 && ask(P, 2) == 2 && calls == c);
    CHECK(ask(P, 9) == 9 && used == 270);  // another, larger term asks anew
  }
  {  // nothing at all
    ImagePool P;
    free_bytes = 0; total_bytes = 1000000; limit = 0; used = 0;
    CHECK(ask(P, 5) == 0 && ask(P, 5) == 0 && used == 0);
  }
  return 0;
}
"""


def test_reserve(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "pool.cpp", tmp_path / "pool"
    src.write_text(SRC)
    subprocess.run([gxx, "-std=c++17", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_1609_02652_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

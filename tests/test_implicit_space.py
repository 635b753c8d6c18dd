"""The implicit solver's work space (csrc/implicit_space.h) is taken together or not at
all: whichever of its requests fails, nothing stays allocated, no size is recorded, and
the next call asks for everything again.  Host code, compiled here with a counting
allocator that fails the request of a given number."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_13487_gb300", "csrc")

PROGRAM = r"""
#include "implicit_space.h"
#include <cstdio>
#include <cstdlib>
#include <set>
using namespace fedbm;
static std::set<void*> live;
static int count = 0, fail_at = -1;
static int take(void** p, size_t bytes) {
  if (count++ == fail_at) return 2;
  *p = std::malloc(bytes ? 1 : 0);
  live.insert(*p);
  return 0;
}
static int take_event(void** p) { return take(p, 1); }
static void give(void* p) {
  if (!live.erase(p)) { std::puts("freed what was not taken"); std::exit(1); }
  std::free(p);
}
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s (request %d)\n", __LINE__, #c, fail_at); std::exit(1); } } while (0)
static bool whole(const ImplicitSpace& s, bool f32) {
  return s.u0 && s.Y && s.base && s.RY && s.G && s.d && s.w && s.Yp && s.Rp && s.V && s.k && s.partial && s.hdev &&
         s.zpart && s.step && s.npart && s.hcol && s.column && s.scratch && s.geo_unit && (!f32 || (s.x32 && s.r32));
}
int main() {
  const SpaceMemory mem = {&take, &take, &take_event, &give, &give, &give};
  bool fresh;
  for (int f32 = 0; f32 < 2; ++f32) {
    const size_t rb = f32 ? 4 : 8;
    ImplicitSpace s;
    count = 0; fail_at = -1;
    CHECK(s.reserve(mem, 100, 30, 3, 8, rb, 64, &fresh) == 0 && fresh && whole(s, f32));
    const int total = count;
    CHECK(total >= 18 && int(live.size()) == total);
    // what is there is kept for the same or smaller sizes
    CHECK(s.reserve(mem, 100, 20, 1, 8, rb, 64, &fresh) == 0 && !fresh && count == total && s.m == 30);
    // larger: each request fails in turn, with the preconditioner's buffers in place
    for (fail_at = 0; fail_at < total; ++fail_at) {
      count = -1000;
      CHECK(s.reserve_blocks(mem, 10, 5, 5, &fresh) == 0);
      count = 0;
      CHECK(s.reserve(mem, 100, 40 + fail_at, 3, 8, rb, 64, &fresh) == 2 && !fresh);
      CHECK(live.empty() && s.n == 0 && s.m == 0 && s.s == 0 && !s.V && !s.hcol && !s.column && !s.minv && !s.fmask);
      const int asked = fail_at;
      fail_at = -1; count = 0;
      CHECK(s.reserve(mem, 100, 40 + asked, 3, 8, rb, 64, &fresh) == 0 && fresh && whole(s, f32) && count == total);
      fail_at = asked;
    }
    for (int q = 0; q < 4; ++q) {
      const size_t before = live.size();
      count = 0; fail_at = q;
      CHECK(s.reserve_blocks(mem, 10, 5, 5, &fresh) == 2 && !fresh);
      CHECK(live.size() == before && !s.minv && !s.z && !s.ops && !s.fmask && s.n == 100);
      fail_at = -1;
      CHECK(s.reserve_blocks(mem, 10, 5, 5, &fresh) == 0 && fresh && s.minv && s.z && s.ops && s.fmask);
      CHECK(s.reserve_blocks(mem, 10, 5, 5, &fresh) == 0 && !fresh);
      s.release_blocks(mem);
    }
    s.release(mem);
    CHECK(live.empty());
  }
  std::puts("ok");
  return 0;
}
"""


def test_every_failed_request_leaves_an_empty_space(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    src = tmp_path / "space.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "space")
    subprocess.run([cxx, "-std=c++17", "-Wall", "-I" + CSRC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


def test_the_solver_takes_its_work_space_from_there_only():
    """No other allocation stands behind the 'already allocated' test."""
    text = open(os.path.join(CSRC, "capi.cu")).read()
    body = text[text.index("int ensure_implicit("):text.index("// r = R(x): one fused")]
    assert "cudaMalloc" not in body and "cudaHostAlloc" not in body and "im.n =" not in body
    assert "im.reserve(" in body and "im.reserve_blocks(" in body

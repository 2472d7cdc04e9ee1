"""CPU test of the posted states of the run-ahead loop (csrc/rid_posted.h) on a stand-in for
the CUDA runtime, in which a copy takes place only when somebody waits for it: a call
that ends between a post and its read must not leave a copy on its way into the slots
that the thread's next call uses.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <thread>
#include <vector>
#include "rid_posted.h"

#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); std::exit(1); } } while (0)

struct Copy { void* dst; const void* src; size_t n; bool done; };
static std::vector<Copy> copies;   // in stream order
static int live_events = 0, live_pinned = 0;
static bool fail_alloc = false, fail_create = false, fail_copy = false, fail_record = false;
static void finish(size_t upto) {
  for (size_t i = 0; i < upto; ++i)
    if (!copies[i].done) {
      std::memcpy(copies[i].dst, copies[i].src, copies[i].n);
      copies[i].done = true;
    }
}
static bool idle() {
  for (const Copy& c : copies)
    if (!c.done) return false;
  return true;
}
struct Rt {
  using Stream = int;
  using Event = size_t;  // copies issued before the record
  static void* alloc_pinned(size_t n) { if (fail_alloc) return nullptr; ++live_pinned; return std::calloc(1, n); }
  static void free_pinned(void* p) { --live_pinned; std::free(p); }
  static bool create(Event*) { if (fail_create) return false; ++live_events; return true; }
  static void destroy(Event) { --live_events; }
  static bool copy(void* d, const void* s, size_t n, Stream) {
    if (fail_copy) return false;
    copies.push_back({d, s, n, false});
    return true;
  }
  static bool record(Event& e, Stream) { if (fail_record) return false; e = copies.size(); return true; }
  static bool wait(Event e) { finish(e); return true; }
  static void wait_stream(Stream) { finish(copies.size()); }
};
struct State { int v; int w; };
using Posted = rid::PostedStates<State, Rt>;

int main() {
  State dev[8];
  for (int i = 0; i < 8; ++i) dev[i] = {10 + i, i};
  State h{};
  {  // one behind: each read gives its own state
    Posted p;
    CHECK(p.open());
    for (int t = 1; t < 6; ++t) {
      CHECK(p.post(t, &dev[t], 0));
      if (t > 1) { CHECK(p.read(t - 1, &h)); CHECK(h.v == 10 + t - 1); }
    }
    CHECK(p.read(5, &h) && h.v == 15);
  }
  CHECK(idle() && live_events == 0);
  {  // given up with two posted
    Posted p;
    CHECK(p.open() && p.post(1, &dev[1], 0) && p.post(2, &dev[2], 0));
  }
  CHECK(idle() && live_events == 0);
  {  // a post on a slot that was not read waits for the copy before it
    Posted p;
    CHECK(p.open() && p.post(1, &dev[1], 0) && p.post(3, &dev[3], 0));
    CHECK(p.read(3, &h) && h.v == 13);
  }
  CHECK(idle());
  {  // no event behind the copy
    Posted p;
    CHECK(p.open());
    fail_record = true;
    CHECK(!p.post(1, &dev[1], 0));
    fail_record = false;
    CHECK(idle());
  }
  {
    Posted p;
    CHECK(p.open());
    fail_copy = true;
    CHECK(!p.post(1, &dev[1], 0));
    fail_copy = false;
  }
  CHECK(idle() && live_events == 0 && live_pinned == 1);
  std::thread([] {  // a thread's slots are its own and go with it
    { Posted p; CHECK(p.open()); }
    CHECK(live_pinned == 2);
  }).join();
  CHECK(live_pinned == 1);
  std::thread([] {
    fail_alloc = true;
    { Posted p; CHECK(!p.open()); }
    fail_alloc = false;
    fail_create = true;
    { Posted p; CHECK(!p.open()); }
    fail_create = false;
  }).join();
  CHECK(live_events == 0 && live_pinned == 1);
  std::puts("ok");
}
"""


def test_posted_states(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "posted.cpp", tmp_path / "posted"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", os.path.join(ROOT, "paper_2310_09417_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout

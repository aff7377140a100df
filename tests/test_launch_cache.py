"""What the host path keeps about its kernels (csrc/launch_cache.h), compiled
for the CPU with a driver made of plain variables: answers for every shape the
library asks about, failed queries asked again, and the shared memory of a
kernel that threads launch with different sizes."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "launch_cache.h"
#include <atomic>
#include <cstdio>
#include <cstring>
#include <thread>
#include <vector>
static sbd::LaunchCache cache;
static const void* fn(int i) { return reinterpret_cast<const void*>((uintptr_t)(0x400000 + 16 * i)); }

static int shapes() {         // every shape of the library twice: one query each, its own answer
  int queries = 0;
  for (int rep = 0; rep < 2; ++rep) {
    int at = 0;
    auto ask = [&](int f, int threads, size_t smem, int cluster) {
      const int want = ++at;
      if (cache.clusters(fn(f), threads, smem, cluster, [&] { ++queries; return want; }) != want) return false;
      return true;
    };
    for (int f = 0; f < 4; ++f)
      for (int c = 2; c <= 16; ++c) if (!ask(f, 320, 230400, c)) return 1;
    for (int f = 4; f < 10; ++f)
      for (int c : {16, 12, 10, 8, 6, 5, 4, 3, 2}) if (!ask(f, 256, 92000, c)) return 2;
    for (int rows = 16; rows <= 160; rows += 16)
      for (int c = 2; c <= 8; ++c) if (!ask(10, 320, 1024 + 2048 * rows, c)) return 3;
    for (int f = 11; f < 17; ++f) if (!ask(f, 320, 228352, 2)) return 4;
    if (!ask(11, 256, 228352, 2)) return 5;          // other threads, another answer
    if (queries != at) return 6;
  }
  return 0;
}

static int failures() {       // an answer < 0 is not kept, one of 0 is
  int n = 0;
  auto bad = [&] { ++n; return -1; };
  auto none = [&] { ++n; return 0; };
  if (cache.clusters(fn(40), 32, 0, 2, bad) != 0 || cache.clusters(fn(40), 32, 0, 2, bad) != 0 || n != 2) return 1;
  if (cache.clusters(fn(40), 32, 0, 2, [&] { ++n; return 7; }) != 7 || cache.clusters(fn(40), 32, 0, 2, bad) != 7) return 2;
  if (cache.clusters(fn(41), 32, 0, 2, none) != 0 || cache.clusters(fn(41), 32, 0, 2, bad) != 0 || n != 4) return 3;
  return 0;
}

static int threads() {        // a launch after its own call finds at least what it asked for
  std::atomic<size_t> limit{0};
  std::atomic<int> short_of{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 4; ++t)
    ts.emplace_back([&, t] {
      const size_t need = 50000 + 10000 * t;
      for (int i = 0; i < 20000; ++i) {
        cache.allow_smem(fn(50), need, [&](size_t most) { limit = most; return 0; });
        if (limit < need) ++short_of;
      }
    });
  for (auto& t : ts) t.join();
  if (short_of != 0) return 1;
  // a refused size is returned and changes nothing
  if (cache.allow_smem(fn(50), 1000000, [](size_t) { return 5; }) != 5) return 2;
  size_t got = 0;
  if (cache.allow_smem(fn(50), 1, [&](size_t most) { got = most; return 0; }) != 0 || got != 80000) return 3;
  return 0;
}

static int full() {           // past its room it asks every time, and stays right
  for (int i = 0; i < 2 * sbd::LaunchCache::kEntries; ++i)
    if (cache.clusters(fn(100 + i), 32, 0, 2, [&] { return i; }) != i) return 1;
  int n = 0;
  for (int rep = 0; rep < 2; ++rep)
    if (cache.clusters(fn(99), 32, 0, 2, [&] { ++n; return 3; }) != 3) return 2;
  return n == 2 ? 0 : 3;
}

int main(int, char** argv) {
  const char* w = argv[1];
  return !strcmp(w, "shapes") ? shapes() : !strcmp(w, "failures") ? failures() : !strcmp(w, "threads") ? threads() : full();
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("launch_cache")
    src, exe = d / "t.cpp", d / "t"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread",
                    "-I" + os.path.join(ROOT, "paper_2509_04185_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("what", ["shapes", "failures", "threads", "full"])
def test_launch_cache(program, what):
    r = subprocess.run([program, what], timeout=60)
    assert r.returncode == 0, (what, r.returncode)

"""The host's parallel set-up loop (host_parallel.h), compiled on its own: every run is done once,
and whichever allocation of the call fails (thread states, the thread list), it either completes or
throws: it never ends the process with threads still running."""
import os
import subprocess

from paper_2202_10313_gb300 import build

PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <new>
#include <stdexcept>
#include "HEADER"
static std::thread::id main_thread;
static long left = -1;   // allocations of the main thread until one fails (-1: none)
void* operator new(std::size_t n) {
  if (left >= 0 && std::this_thread::get_id() == main_thread && left-- == 0) throw std::bad_alloc();
  if (void* p = std::malloc(n)) return p;
  throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
int main() {
  main_thread = std::this_thread::get_id();
  const int64_t n = 1003;
  static std::atomic<int> hits[n];
  auto fn = [&](int64_t b, int64_t e) { for (; b < e; ++b) hits[b]++; };
  for (long k = -1; k < 40; ++k) {
    for (auto& h : hits) h = 0;
    bool threw = false;
    left = k;
    try { lts::host_parallel(n, 10, fn, 16); } catch (const std::bad_alloc&) { threw = true; }
    left = -1;
    for (auto& h : hits) if (h != (threw ? 0 : 1)) return 1;
    if (k < 0 && threw) return 2;
  }
  bool caught = false;
  try {
    lts::host_parallel(n, 10, [&](int64_t b, int64_t) { if (b > n / 2) throw std::runtime_error("x"); }, 16);
  } catch (const std::runtime_error&) { caught = true; }
  if (!caught) return 3;
  std::puts("ok");
}
"""


def test_a_failed_allocation_never_ends_the_process(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM.replace("HEADER", os.path.join(build.SRC, "host_parallel.h")))
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert (r.returncode, r.stdout.strip()) == (0, "ok"), (r.returncode, r.stderr)

"""The parts of the library that are plain C++ headers, compiled and run on the CPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_18893_b200", "csrc")


@pytest.fixture
def run_cpp(tmp_path):
    def run(source):
        src, exe = tmp_path / "t.cpp", tmp_path / "t"
        src.write_text(source)
        subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
        r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
        assert r.returncode == 0, r.stdout + r.stderr
    return run


def test_a_limit_is_never_recorded_above_what_is_set(run_cpp):
    """Two threads' first calls: the larger size is set, and before that is on record the other thread asks for less."""
    run_cpp(r"""
#include <chrono>
#include <cstdio>
#include <thread>
#include "xkv_grow.h"
int main() {
  std::atomic<size_t> have{0}, set_to{0};
  std::mutex lock;
  std::atomic<bool> large_is_set{false};
  std::atomic<int> calls{0};
  std::thread small([&] {
    while (!large_is_set) std::this_thread::yield();
    xkv::grow(have, lock, 160, [&](size_t to) { ++calls; set_to = to; return 0; });
  });
  xkv::grow(have, lock, 192, [&](size_t to) {
    ++calls; set_to = to; large_is_set = true;
    std::this_thread::sleep_for(std::chrono::milliseconds(200));
    return 0;
  });
  small.join();
  if (set_to < have || have != 192 || calls != 1) { printf("set %zu, on record %zu, %d calls\n", set_to.load(), have.load(), calls.load()); return 1; }
  // a failure leaves the record alone and is handed on; the next call tries again
  if (xkv::grow(have, lock, 200, [](size_t) { return 7; }) != 7 || have != 192) return 2;
  if (xkv::grow(have, lock, 200, [&](size_t to) { set_to = to; return 0; }) != 0 || have != 200 || set_to != 200) return 3;
  return 0;
}
""")


def test_the_gather_from_codes_stays_inside_the_row(run_cpp):
    """Every rank up to 8192, the largest of a handle, every pair of slabs, every lane; and every group
    of the row is fetched, by the lane whose columns it holds."""
    run_cpp(r"""
#include <cstdio>
#include "xkv_gather.h"
int main() {
  for (int rank = 32; rank <= 8192; rank += 32) {
    const int groups = rank / 32, slabs = ((rank + 63) / 64 + 1) & ~1;     // slabs are padded to pairs
    int fetched[256] = {};
    for (int ks = 0; ks < slabs; ks += 2)
      for (uint32_t lane = 0; lane < 4; ++lane) {
        const uint32_t at = xkv::quant_group(ks, lane, rank);
        if (at >= (uint32_t)groups) { printf("rank %d, slab %d, lane %u: group %u\n", rank, ks, lane, at); return 1; }
        if (ks * 64 + (int)lane * 32 == (int)at * 32) ++fetched[at];
      }
    for (int i = 0; i < groups; ++i) if (fetched[i] != 1) { printf("rank %d: group %d fetched %d times\n", rank, i, fetched[i]); return 1; }
  }
  return 0;
}
""")

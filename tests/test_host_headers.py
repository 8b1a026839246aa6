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

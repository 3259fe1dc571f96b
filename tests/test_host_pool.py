"""The host threads of the library's copies (csrc/host_pool.h), as a program of
their own: every part of a job runs once, and a caller that finds the workers
busy does not wait for them."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(__file__)), "paper_1712_03560_gb300", "csrc")

PROGRAM = r"""
#include <chrono>
#include <cstdio>

#include "host_pool.h"

using namespace oasm;

static bool every_part_once(size_t n, size_t least) {
  std::vector<std::atomic<int>> seen(n);
  parallel_parts(n, least, [&](size_t lo, size_t hi) {
    for (size_t i = lo; i < hi; ++i) seen[i] += 1;
  });
  for (auto& s : seen)
    if (s != 1) return false;
  return true;
}

int main() {
  for (size_t n : {0, 1, 15, 16, 17, 100000})
    for (size_t least : {1, 16, 200000})
      if (!every_part_once(n, least)) return 1;
  // one caller's job goes on until another caller's has ended
  std::atomic<bool> started{false}, other{false};
  bool waited = false;
  std::thread first([&] {
    const std::function<void(size_t)> job = [&](size_t i) {
      if (i) return;
      started = true;
      const auto end = std::chrono::steady_clock::now() + std::chrono::seconds(3);
      while (!other && std::chrono::steady_clock::now() < end) std::this_thread::yield();
      waited = !other;
    };
    HostPool::get().run(4, job);
  });
  while (!started) std::this_thread::yield();
  const bool all = every_part_once(100000, 1);
  other = true;
  first.join();
  return !all ? 2 : waited ? 3 : 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_callers_do_not_wait_for_one_another(tmp_path):
    src, exe = tmp_path / "pool.cpp", tmp_path / "pool"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    assert subprocess.run([str(exe)], timeout=60).returncode == 0

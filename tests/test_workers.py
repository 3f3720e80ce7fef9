"""The SPMD harnesses' kept threads (csrc/gvm_workers.h) on the CPU."""
import os
import shutil
import signal
import subprocess

import pytest

from conftest import ROOT

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>

#include "gvm_workers.h"

int main(int argc, char** argv) {
  gvm::WorkerPool pool;
  if (argc > 1 && !strcmp(argv[1], "throw")) {
    try {
      pool.run(4, [](int r) {
        if (r == 0) throw std::bad_alloc();
        std::this_thread::sleep_for(std::chrono::milliseconds(200));
      });
    } catch (...) {
      printf("unwound with workers running\n");
      fflush(stdout);
      _Exit(3);
    }
    return 4;
  }
  // Runs of changing width, back to back and after the workers fell asleep,
  // and two at once: every rank of every run exactly once.
  auto check = [&](int n) {
    std::vector<std::atomic<int>> seen(n);
    for (auto& s : seen) s = 0;
    if (pool.run(n, [&](int r) { seen[r].fetch_add(1); }) != GVM_OK) return false;
    for (auto& s : seen)
      if (s != 1) return false;
    return true;
  };
  for (int i = 0; i < 300; ++i) {
    if (!check(1 + (i * 7) % 13)) return 1;
    if (i % 50 == 0) std::this_thread::sleep_for(std::chrono::milliseconds(2));
  }
  bool other = true;
  std::thread t([&] {
    for (int i = 0; i < 200; ++i) other = check(1 + i % 5) && other;
  });
  bool mine = true;
  for (int i = 0; i < 200; ++i) mine = check(1 + i % 7) && mine;
  t.join();
  return mine && other ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("workers")
    (d / "w.cpp").write_text(PROGRAM)
    exe = str(d / "w")
    r = subprocess.run([gxx, "-O2", "-std=c++17", "-Wall", "-Werror", "-pthread",
                        "-I", os.path.join(ROOT, "paper_1511_07658_gb300", "csrc"),
                        "-I", os.path.join(ROOT, "include"), str(d / "w.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


def test_every_rank_runs_once(program):
    assert subprocess.run([program], timeout=120).returncode == 0


def test_exception_of_the_calling_rank_ends_the_program(program):
    # As one on a thread of its own does; it must not unwind the frame that the other ranks still use.
    r = subprocess.run([program, "throw"], capture_output=True, text=True, timeout=60)
    assert r.returncode == -signal.SIGABRT, (r.returncode, r.stdout)

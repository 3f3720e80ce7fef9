"""The pair form's k-step numbering (csrc/gvm_ring.h), walked on the CPU from a
launch's first tile past 2^32 k-steps, as a resident scheduler passes it: every
k-step's stage, barrier, phase parity and group must be those of a counter that
never wraps. The same walk with a plain 32-bit counter must not pass, so that
the walk is known to see the fault."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

PROGRAM = r"""
#include <stdio.h>

#include "gvm_ring.h"
using namespace gvm;

// q stands for k-step Q of a launch, both for the waits and for the arrivals.
static bool same(uint32_t q, uint64_t Q) {
  return pr_stage(q) == Q % 3 && pr_full_parity(q) == ((Q / 3) & 1) && pr_empty_bar(q) == Q % 6 &&
         pr_empty_parity(q) == ((Q / 6) & 1) && (q & 1) == (Q & 1) && pr_stage_used(q) == (Q >= 3) &&
         (Q < 3 || (pr_empty_bar(q - 3) == (Q - 3) % 6 && pr_empty_parity(q - 3) == (((Q - 3) / 6) & 1)));
}

int main() {
  const uint64_t end = (1ull << 32) + 20000;
  uint64_t Q = 0, plain_wrong = 0;
  uint32_t first = 0, seed = 1;
  while (Q < end) {
    seed = seed * 1664525u + 1013904223u;
    // Tiles of one to four k-steps at the launch's start and around 2^32, up to 1024 (k = 32768) between.
    const bool edge = Q < 20000 || Q > (1ull << 32) - 20000;
    const uint32_t ksteps = 1 + (seed >> 8) % (edge ? 4 : 1024);
    for (uint32_t i = 0; i < ksteps; i += edge ? 1 : 97) {
      if (!same(first + i, Q + i)) {
        printf("k-step %llu of the launch, numbered %u\n", (unsigned long long)(Q + i), first + i);
        return 1;
      }
      if (!same((uint32_t)(Q + i), Q + i)) ++plain_wrong;
    }
    first = pr_next_first(first, ksteps);
    Q += ksteps;
  }
  printf("%llu\n", (unsigned long long)plain_wrong);
  return 0;
}
"""


def test_numbering_holds_past_2_to_32_ksteps(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "ring.cpp", tmp_path / "ring"
    src.write_text(PROGRAM)
    inc = os.path.join(ROOT, "paper_1511_07658_gb300", "csrc")
    r = subprocess.run([gxx, "-O2", "-std=c++17", "-Wall", "-Werror", "-I", inc, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 1000  # a counter left to wrap goes wrong

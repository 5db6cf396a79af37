"""The staging arena (csrc/gbs_stage.h): bytes whose asynchronous copy may still be queued are not
written again before a wait, also across calls that end without one (a sampler step).  Compiled
and run on the host."""
import subprocess
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_1810_00900_gb300" / "csrc"

HARNESS = r"""
#include "gbs_stage.h"
#include <stdio.h>
#include <stdlib.h>
#include <utility>
#include <vector>
using gbs::StageArena;
int main() {
  srand(1);
  long waits = 0, takes = 0;
  for (int trial = 0; trial < 2000; ++trial) {
    StageArena a;
    a.cap = 4096 + 256 * (rand() % 64);
    std::vector<std::pair<size_t, size_t>> queued;  // regions staged since the last wait
    auto wait = [&] { queued.clear(); a.waited(); ++waits; };
    for (int call = 0; call < 20; ++call) {
      if (a.begin()) {
        wait();
        if (a.begin()) return printf("begin() after a wait asks for another\n"), 1;
      }
      const int n = rand() % 8;
      for (int i = 0; i < n; ++i) {
        const size_t bytes = rand() % (rand() % 4 ? 300 : 3000);
        if (!a.fits(bytes)) break;
        if (!a.clear(bytes)) wait();
        const size_t at = a.take(bytes);
        ++takes;
        if (at % 256 || at + bytes > a.cap) return printf("outside the arena\n"), 1;
        for (auto& q : queued)
          if (at < q.first + q.second && q.first < at + bytes) return printf("overwrites a queued copy\n"), 1;
        if (bytes) queued.emplace_back(at, bytes);
        if (rand() % 3 == 0) wait();
      }
      if (rand() % 2) wait();  // other calls end with copies still queued
    }
  }
  // a sampler step: trees, wait, decisions, wait, conditioning; the next step needs no more waits
  StageArena a;
  a.cap = 1 << 20;
  for (int step = 0; step < 3; ++step) {
    if (a.begin()) return printf("a step waits at its start\n"), 1;
    for (size_t bytes : {4000, 9000}) {
      if (!a.clear(bytes)) return printf("a step waits for the one before\n"), 1;
      a.take(bytes);
    }
    a.waited();
    a.take(3000);
    a.waited();
    a.take(2000);
  }
  printf("ok %d\n", takes > 10000 && waits > 1000);
  return 0;
}
"""


def test_no_region_is_written_while_its_copy_may_be_queued(tmp_path):
    src, exe = tmp_path / "stage.cpp", tmp_path / "stage"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-I", str(CSRC), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout == "ok 1\n", r.stdout

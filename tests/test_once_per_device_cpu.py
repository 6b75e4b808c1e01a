"""The dynamic shared memory a kernel opts into is set on every device that is
used, not once per process, and a failure is tried again: csrc/ff_once.h
against a fake of the two CUDA calls, and no other way of setting it in the
sources."""

import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_08573_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "ff_once.h"
enum Status { OK, FAIL };
int main() {
  std::atomic<unsigned long long> done{0};
  std::atomic<int> calls[65] = {};
  thread_local static int current = 0;
  bool broken = false;
  auto get = [](int* d) { *d = current; return OK; };
  auto set = [&] { ++calls[current]; return broken ? FAIL : OK; };
  auto call = [&] { return ff::once_per_device<Status>(done, get, set); };
  bool good = call() == OK && call() == OK && calls[0] == 1;
  current = 1;                                     // a second device
  broken = true;
  good = good && call() == FAIL && call() == FAIL && calls[1] == 2;
  broken = false;                                  // a failure is not kept
  good = good && call() == OK && call() == OK && calls[1] == 3;
  current = 64;                                    // past the bits: every time
  good = good && call() == OK && call() == OK && calls[64] == 2;
  std::vector<std::thread> t;
  for (int i = 0; i < 8; ++i) t.emplace_back([&, i] { current = 2 + i % 4; for (int k = 0; k < 1000; ++k) call(); });
  for (auto& x : t) x.join();
  for (int d = 2; d < 6; ++d) good = good && calls[d] >= 1 && calls[d] <= 2;
  std::puts(good ? "good" : "bad");
}
"""


def test_once_per_device(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, timeout=60).stdout.strip() == "good"


def test_kernels_set_their_shared_memory_through_it():
    for f in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, f)) as h:
            n = len(re.findall(r"cudaFuncSetAttribute\(", h.read()))
        assert n == (1 if f == "ff_internal.cuh" else 0), f

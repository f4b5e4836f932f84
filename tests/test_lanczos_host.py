"""Host side of the truncation that needs no GPU, compiled with g++ against a
stream whose copies read their source only when it is waited for (CUDA lets a
copy from pageable memory do so)."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2602_20376_gb300", "csrc")


def _run(tmp_path, body):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(body)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


def test_copies_outlive_the_stream(tmp_path):
    out = _run(tmp_path, r"""
#include <cstdio>
#include <cstring>
#include "lanczos_host.h"
struct Copy { double* to; const double* from; int n; };
static std::vector<Copy> queue;
static void wait_stream() {
  for (const Copy& c : queue) std::memcpy(c.to, c.from, c.n * sizeof(double));
  queue.clear();
}
static double dev[64][1000];
static int drive(int rounds, bool fail) {
  auto wait = []() { wait_stream(); };
  lrq::HostCopies<decltype(wait)> copies(wait);
  for (int k = 0; k < rounds; ++k) {
    std::vector<double> x(1000, k + 0.5);
    const int n = static_cast<int>(x.size());
    queue.push_back(Copy{dev[k], copies.keep(std::move(x)), n});
    std::vector<double> other(1000, -1.0);  // takes a freed block's place
    if (fail && k == rounds / 2) return 1;
  }
  return 0;
}
int main() {
  int bad = 0;
  for (int fail = 0; fail < 2; ++fail) {
    std::memset(dev, 0, sizeof(dev));
    drive(64, fail);
    for (int k = 0; k < (fail ? 33 : 64); ++k)
      for (int i = 0; i < 1000; ++i) bad += dev[k][i] != k + 0.5;
  }
  std::printf("%d %d\n", bad, static_cast<int>(queue.size()));
}
""")
    assert out == ["0", "0"]


def test_every_copy_from_the_host_is_kept():
    # the truncation's host-to-device copies read what the holder keeps
    text = open(os.path.join(CSRC, "k_lanczos.cu")).read()
    calls = re.findall(r"cudaMemcpyAsync\(([^;]*?)cudaMemcpyHostToDevice", text, re.S)
    assert calls and all("copies.keep(" in c for c in calls)

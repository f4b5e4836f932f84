"""Host side of the truncation that needs no GPU, compiled with g++ against a
stream whose copies read their source only when it is waited for (CUDA lets a
copy from pageable memory do so)."""
import os
import re
import shutil
import subprocess

import numpy as np
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


@pytest.mark.parametrize("nc", [1, 8, 156, 500, 4096])
@pytest.mark.parametrize("cplx", [False, True])
def test_fp32_correction_moves_w_by_a_rounding(tmp_path, nc, cplx):
    """The FP32 chain of lz_update at the largest h its gate lets through, on the
    entries of random unit vectors: below 2^-52 ||w|| (||w|| = 1)."""
    body = '#include <cstdio>\n#include "lanczos_host.h"\nint main() { std::printf("%%a", lrq::lz_fp32_gate(%d)); }'
    gate = float.fromhex(_run(tmp_path, body % nc)[0])
    n, f32 = 2048, np.float32
    g = np.random.Generator(np.random.PCG64(nc))

    def cut(x):  # to FP32, towards zero
        y = x.astype(f32)
        return np.where(np.abs(y.astype(np.float64)) > np.abs(x), np.nextafter(y, f32(0)), y)

    def fma(a, b, c):  # the product of two FP32 numbers is exact in FP64, the sum rounds to FP32 after one of 2^-53
        return (a.astype(np.float64) * np.float64(b) + c.astype(np.float64)).astype(f32)

    parts = 2 if cplx else 1
    h = g.standard_normal((nc, parts))
    h *= gate / np.abs(h).sum()  # sum |Re h_c| + |Im h_c| at the gate
    exact, t = np.zeros((n, parts)), np.zeros((n, parts), f32)
    for c in range(nc):
        u = g.standard_normal((n, parts))
        u /= np.linalg.norm(u)
        uf, hf = cut(u), cut(h[c])
        if cplx:
            exact += np.stack([u[:, 0] * h[c, 0] - u[:, 1] * h[c, 1], u[:, 0] * h[c, 1] + u[:, 1] * h[c, 0]], 1)
            re = fma(uf[:, 0], hf[0], fma(-uf[:, 1], hf[1], t[:, 0]))
            im = fma(uf[:, 0], hf[1], fma(uf[:, 1], hf[0], t[:, 1]))
            t = np.stack([re, im], 1)
        else:
            exact += u * h[c]
            t = fma(uf, hf[0], t)
    assert np.linalg.norm(t - exact) <= 2.0 ** -52
    # and with every rounding against it
    roundings = (2 if cplx else 1) * nc + 12
    assert roundings * 2.0 ** -24 * gate <= 2.0 ** -52

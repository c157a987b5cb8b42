"""Host checks of the triangular normal basis (no GPU): a small program is compiled against the plan and
the kernel header.  For every degree and several sets of weights, B diag(D) B^T must reproduce
sum_j c_j g_j g_j^T and B must have the unit and zero entries that the face kernel takes for granted
(Pivots<K>); the benchmark's flop count uses the same pivots.  Weights without a usable basis (negative, NaN,
infinite, factors at the ends of the range) must have none, so that the jump vectors themselves run and
the result is what those weights give."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_00246_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <limits>
#include <utility>
#include <vector>
#include "gp_kernels.cuh"
#include "gp_plan.h"

int bad = 0;
void fail(const char* what, int k, int kind) { std::printf("FAIL %s k=%d weights %d\n", what, k, kind); ++bad; }

template <int K>
void check() {
  constexpr int N = K + 1, NN = 2 * K + 1;
  std::vector<double> gl, mass, g, ldl;
  std::vector<long double> D;
  gp::gauss_lobatto_01(K, gl);
  gp::reference_1d(K, gl, mass, g);
  const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
  for (int kind = 0; kind < 5; ++kind) {
    std::vector<double> c(K, 0.5);
    double f = 1.0;
    for (int j = 0; j < K; ++j) {
      f *= j + 1;
      if (kind == 1) c[j] = 0.5 / (f * f);
      if (kind == 2) c[j] = j == 0 ? 0.5 : 0.0;
      if (kind == 3) c[j] = j == K - 1 ? 0.5 : 0.0;
      if (kind == 4) c[j] = 0.0;
    }
    const double hd = 0.03125;
    gp::normal_basis(K, g, c, hd, ldl, D);
    if (ldl.size() != (size_t)(K * N) || D.size() != (size_t)K) { fail("no basis", K, kind); continue; }
    auto B = [&](int j, int b) -> double {          // row j on the folded line, mirrored with its parity
      return b <= K ? ldl[j * N + b] : (j & 1 ? -1.0 : 1.0) * ldl[j * N + NN - 1 - b];
    };
    long double top = 0;
    for (int b = 0; b < NN; ++b) {
      long double s = 0;
      for (int j = 0; j < K; ++j) s += (long double)c[j] * g[j * NN + b] * g[j * NN + b];
      top = std::max(top, hd * s);
    }
    for (int a = 0; a < NN; ++a)
      for (int b = 0; b < NN; ++b) {
        long double s = 0, t = 0;
        for (int j = 0; j < K; ++j) {
          s += (long double)hd * c[j] * g[j * NN + a] * g[j * NN + b];
          t += D[j] * B(j, a) * B(j, b);
        }
        // every entry and every factor is rounded once: a few units in the last place of the largest entry
        if (!(std::fabs((double)(s - t)) <= 4 * K * 1.2e-16L * top)) { fail("B D B^T", K, kind); a = b = NN; }
      }
    for (int j = 0; j < K; ++j) {
      if (B(j, gp::Pivots<K>::at(j)) != 1.0) fail("pivot entry", K, kind);
      for (int b = 0; b <= K; ++b)
        if (gp::Pivots<K>::zero(j, b) && B(j, b) != 0.0) fail("zero entry", K, kind);
      if ((j & 1) && B(j, K) != 0.0) fail("odd row at the face", K, kind);
      if (!(D[j] >= 0.0)) fail("factor", K, kind);
    }
  }
  const double none[] = {inf, nan, -0.5, -inf, 1e300, 1e-305};
  for (int kind = 0; kind < 6; ++kind)
    for (int j = 0; j < K; ++j) {
      std::vector<double> c(K, kind >= 4 ? none[kind] : 0.5);
      c[j] = none[kind];
      gp::normal_basis(K, g, c, 0.03125, ldl, D);
      if (!ldl.empty()) fail("basis of unusable weights", K, 10 + kind);
    }
  std::printf("%d:", K);
  for (int j = 0; j < K; ++j) std::printf(" %d", gp::Pivots<K>::at(j));
  std::printf("\n");
}

template <int... Ks>
void all(std::integer_sequence<int, Ks...>) { (check<Ks + 1>(), ...); }

int main() {
  all(std::make_integer_sequence<int, 8>{});
  return bad ? 1 : 0;
}
"""


def _nvcc():
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc")):
        if c and os.path.exists(c):
            return c
    return None


def test_triangular_basis(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    src = tmp_path / "basis.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "basis"
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src), os.path.join(CSRC, "gp_plan.cpp"),
                    os.path.join(CSRC, "gp_brick_plan.cpp"), "-o", str(exe)], check=True, capture_output=True, timeout=300)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stdout + out.stderr
    import bench
    piv = {int(line.split(":")[0]): tuple(map(int, line.split(":")[1].split())) for line in out.stdout.split("\n") if line}
    assert piv == bench._PIVOTS

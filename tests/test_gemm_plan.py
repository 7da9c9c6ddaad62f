"""The choice of tile, split and path of the FP64 products (csrc/gemm_plan.cuh), on the
host: over sizes up to outputs of many million elements every product has a plan with a
finite time whose grid and partials are within their limits, nothing below 2e8 flops
leaves the FP64 pipe, and the shapes of test_gpu_gemm_tiles.py reach every tile there."""
import shutil
import subprocess

import pytest

from tests.test_df_arith import CSRC
from tests.test_gpu_gemm_tiles import SHAPES

PROG = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "gemm_plan.cuh"
using namespace pwh;
int main(int argc, char**) {
  int M, N, K;
  if (argc > 1) {
    while (std::scanf("%d %d %d", &M, &N, &K) == 3)
      std::printf("%d %d %d\n", plan64(M, N, K, false).shape, plan64(M, N, K, false).split, (int)oz_wins(M, N, K));
    return 0;
  }
  std::mt19937_64 g(5);
  auto logu = [&](double lo, double hi) {
    std::uniform_real_distribution<double> u(std::log2(lo), std::log2(hi));
    return (int)std::exp2(u(g));
  };
  for (int i = 0; i < 200000; ++i) {
    M = logu(1, 8e6), K = logu(1, 1e6);
    N = logu(1, std::max(2.0, std::min(4e6, 1e9 / M)));
    const Plan64 p = plan64(M, N, K, i & 1);
    const int BM = kShape64[p.shape][0], BN = kShape64[p.shape][1];
    const bool ok = p.us < 1e12 && (N + BN - 1) / BN <= 65535 &&
                    (p.split == 1 || (p.split <= 256 && (double)p.split * M * N * 16 <= 64.0 * (1 << 20))) &&
                    (8.0 * M * N * K >= 2e8 || !oz_wins(M, N, K));
    if (!ok) return std::printf("%d %d %d: %d x %d, split %d, %g us\n", M, N, K, BM, BN, p.split, p.us), 1;
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(PROG)
    subprocess.run([gxx, "-std=c++17", "-O2", "-I", CSRC, str(d / "plan.cpp"), "-o", str(d / "plan")],
                   check=True, timeout=120)
    return str(d / "plan")


def test_every_product_has_a_plan(exe):
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


def test_gpu_shapes_reach_every_tile(exe):
    r = subprocess.run([exe, "s"], input="".join(f"{m} {n} {k}\n" for m, n, k in SHAPES), capture_output=True,
                       text=True, check=True, timeout=60)
    rows = [tuple(map(int, l.split())) for l in r.stdout.splitlines()]
    assert {s for s, _, _ in rows} == set(range(7))
    assert any(p > 1 for _, p, _ in rows) and not any(w for _, _, w in rows)

"""Pieces, segments and workspace of the residue GEMM (csrc/gemm_mod_geom.cuh), on the
host: over sizes up to the largest that the dispatch sends there (65,535 columns, and rows
of A^H; tall A B; K to 2^21), every piece stays within the two fixed caps plus its
norms, covers K with whole 64-wide blocks, and a workspace of mod_bound(M, N, K) holds
every piece of every product of at most M x N x K (what a solver reserves before its
iterations)."""
import shutil
import subprocess

import pytest

from tests.test_df_arith import CSRC

PROG = r"""
#include <cstdio>
#include <random>
#include "gemm_mod_geom.cuh"
using namespace pwh;
static std::mt19937_64 g(7);
static int logu(double hi) {
  std::uniform_real_distribution<double> u(0.0, std::log2(hi + 1.0));
  return std::max(1, (int)std::min(hi, std::exp2(u(g)) - 0.5));
}
static size_t largest = 0;
// the largest workspace of the pieces of a product; 0: a piece is wrong
static size_t need(bool cj, int M, int N, int K) {
  const ModSplit sp = mod_split(cj, M, N, K);
  if (sp.pm < 1 || sp.pn < 1 || sp.pm > M || sp.pn > N) return 0;
  size_t most = 0;
  for (int m : {sp.pm, M % sp.pm ? M % sp.pm : sp.pm})
    for (int n : {sp.pn, N % sp.pn ? N % sp.pn : sp.pn}) {
      const ModGeom q = mod_geom(cj, m, n, K, 76);
      const int per = cj ? 1 : 2;
      if ((int64_t)q.kseg * q.nseg < K || (int64_t)q.kseg * (q.nseg - 1) >= K) return 0;
      if (q.seg % 64 || q.seg < (int64_t)q.kseg * per || (int64_t)q.kb_per * q.gz < q.kb ||
          (int64_t)q.kb_per * (q.gz - 1) >= q.kb) return 0;
      if (q.bn > 256 || q.bn % 32 || q.Np < q.Nr || (int64_t)q.gm * 256 < q.Mr) return 0;
      if (q.bytes_a + q.bytes_b > kOzOperandCap + 512 || q.bytes_r > kOzResidueCap) return 0;
      most = std::max(most, q.total());
    }
  largest = std::max(largest, most);
  return most;
}
int main() {
  const int fixed[][3] = {{161235, 544, 298}, {161235, 544, 544}, {161235, 544, 1632}, {1632, 1632, 161235},
                          {4096, 4096, 161235}, {4096, 4096, 1000000}, {600000, 1000, 16}, {1500, 1500, 2000000},
                          {65535, 65535, 2097120}, {65535, 1, 1}, {1, 65535, 960}, {128, 128, 961}};
  for (int cj = 0; cj < 2; ++cj) {
    for (auto& f : fixed) {
      if (cj && f[0] > 65535) continue;
      const size_t n = need(cj, f[0], f[1], f[2]), b = mod_bound(cj, f[0], f[1], f[2]);
      if (!n || n > b) return std::printf("%d %d %d %d needs %zu of %zu\n", cj, f[0], f[1], f[2], n, b), 1;
    }
    for (int i = 0; i < 20000; ++i) {
      const int M = logu(cj ? 65535 : 5e6), N = logu(65535), K = logu(2097120);
      const size_t b = mod_bound(cj, M, N, K);
      for (int j = 0; j < 4; ++j) {
        const int m = j ? logu(M) : M, n = j ? logu(N) : N, k = j ? logu(K) : K;
        const size_t w = need(cj, m, n, k);
        if (!w || w > b)
          return std::printf("%d: %d %d %d needs %zu, %d %d %d reserves %zu\n", cj, m, n, k, w, M, N, K, b), 1;
      }
    }
  }
  std::printf("%zu\n", largest);
  return 0;
}
"""


def test_workspace_is_bounded_and_reservations_hold(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    src = tmp_path / "geom.cpp"
    src.write_text("#include <cmath>\n" + PROG)
    out = tmp_path / "geom"
    subprocess.run([gxx, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(out)], check=True, timeout=120)
    r = subprocess.run([str(out)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
    # the caps, and norms of at most 264 bytes for each row and column of a piece
    assert int(r.stdout) <= (4 << 30) + (512 << 20)

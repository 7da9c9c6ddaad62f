// Choice of the FP64 product's path and tile by a cost model (gemm.cu).  Host
// arithmetic only.
#pragma once
#include <algorithm>
#include <cstdint>

namespace pwh {

// Products of at least this many flops (8 M N K) may take the tensor cores; smaller
// ones keep FP64 arithmetic element by element (the residue form's error is relative to
// the operands' norms).
constexpr double kOzMinFlops = 2e8;

// Tile and split-K of an FP64 product on the FP64 pipe: the least modelled
// clocks, waves of blocks over 152 SMs times a block's multiply-adds (four a
// complex pair at the measured 1.6 a clock of an SM) and 1,200 clocks of latency,
// plus the reduction of the partials (of a split below 64 MB).  A tile much larger
// than the product computes padding, and few tiles leave the pipe of most SMs
// idle: 32 x 16 over K = 1503 took 176 us in 256 x 16 tiles and takes 20, 1503 x 16
// over K = 32 139 us on six of them and takes 14.
struct Plan64 {
  int shape, split;
  double us;  // modelled time
};
constexpr int kShape64[7][2] = {{64, 64}, {128, 32}, {256, 16}, {256, 8}, {32, 32}, {32, 16}, {16, 16}};
inline Plan64 plan64(int M, int N, int K, bool part) {
  Plan64 best{0, 1, 1e300};
  for (int i = 0; i < 7; ++i) {
    const int BM = kShape64[i][0], BN = kShape64[i][1];
    const int64_t gm = ((int64_t)M + BM - 1) / BM, gn = ((int64_t)N + BN - 1) / BN, tiles = gm * gn;
    if (gn > 65535 && i > 0) continue;  // the grid's y
    for (int w = 0; w <= 6; ++w) {
      int split = w == 0 ? 1 : (int)((152 * (int64_t)w + tiles - 1) / tiles);
      split = std::max(1, std::min(split, std::min(256, K / 16)));
      if (split > 1 && (double)split * M * N * 16.0 > 64.0 * (1 << 20)) continue;
      const int chunk = (((K + split - 1) / split) + 15) / 16 * 16;
      split = std::max(1, (K + chunk - 1) / std::max(chunk, 1));
      const double waves = (double)((tiles * split + 151) / 152);
      double clk = waves * (2.5 * BM * BN * chunk + 1200.0);
      if (split > 1 || part) clk += 5000.0 + split * (double)M * N * 32.0 / 3000.0;
      if (clk < best.us) best = {i, split, clk};
    }
  }
  best.us /= 2000.0;  // 2 GHz
  return best;
}

// Whether an FP64 product goes to the tensor cores (oz_gemm): at least
// kOzMinFlops, and the modelled time there is the smaller: about 40 us of launches
// and latency, the operands read twice and written as 64 bytes a complex number
// (5 TB/s), 128 tensor operations a complex multiply-add (1.2 PFLOP/s), the result.
inline bool oz_wins(int M, int N, int K) {
  if (8.0 * M * (double)N * K < kOzMinFlops) return false;
  const double oz = 40.0 + ((double)M + N) * K * 96.0 / 5e6 + 128.0 * M * (double)N * K / 1.2e9 +
                    (double)M * N * 80.0 / 3e6;
  return oz < plan64(M, N, K, false).us;
}

}  // namespace pwh

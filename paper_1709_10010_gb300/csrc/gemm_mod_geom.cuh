// Geometry and workspace of the residue GEMM (gemm_mod.cu): pieces of the output,
// K segments, K ranges.  Host arithmetic only.
//
// The workspace of a product of any size stays within two fixed parts: the operand
// residues of one K segment (kOzOperandCap) and the residues of the result of one
// piece (kOzResidueCap), which every segment adds to modulo p.  Every choice gives
// the bits of the whole product: the exponents belong to single rows and columns,
// and residues add exactly.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace pwh {

constexpr int kMod = 16;  // moduli
constexpr size_t kOzOperandCap = (size_t)3 << 30;
constexpr size_t kOzResidueCap = (size_t)1 << 30;

inline int64_t oz_round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }
inline size_t oz_align(size_t x) { return (x + 255) & ~(size_t)255; }

// Output tiles of a piece: the fewest of at most 256 columns, all of the least
// width.
struct ModTiles {
  int64_t Mr, Nr, Np;  // real rows and columns, columns of the tiles
  int bn, gm, gn;
};
inline ModTiles mod_tiles(bool conjA, int M, int N) {
  ModTiles t;
  t.Mr = conjA ? 2 * (int64_t)M : M;
  t.Nr = 2 * (int64_t)N;
  t.gm = (int)((t.Mr + 255) / 256);
  t.gn = (int)((t.Nr + 255) / 256);
  t.bn = (int)oz_round_up((t.Nr + t.gn - 1) / t.gn, 32);
  t.Np = (int64_t)t.gn * t.bn;
  return t;
}

struct ModGeom : ModTiles {
  int kseg;       // complex K per segment
  int nseg;
  int64_t seg;    // real K of a segment, padded to 64
  int kb, kb_per, gz;  // 64-wide K blocks, blocks a range, ranges
  int Sa, Sb;     // blocks per row norm
  size_t bytes_a, bytes_b, bytes_r, bytes_n, bytes_e;
  size_t total() const { return bytes_a + bytes_b + bytes_r + bytes_n + bytes_e; }
};
// pairs: CTA pairs resident at once
inline ModGeom mod_geom(bool conjA, int M, int N, int K, int pairs) {
  ModGeom g;
  (ModTiles&)g = mod_tiles(conjA, M, N);
  const int per = conjA ? 1 : 2;  // real K per complex K
  // segments of whole exact chunks (960) whose operand residues fit
  int64_t kmax = (int64_t)(kOzOperandCap / (2 * kMod)) / (g.Mr + g.Nr) / per;
  kmax = std::max<int64_t>(kmax / 960 * 960, 960);
  g.nseg = (int)((K + kmax - 1) / kmax);
  g.kseg = (int)std::min<int64_t>(K, oz_round_up((K + g.nseg - 1) / g.nseg, 64));
  g.nseg = (K + g.kseg - 1) / g.kseg;
  g.seg = oz_round_up((int64_t)g.kseg * per, 64);
  g.kb = (int)(g.seg / 64);
  // K ranges: the count with the least modelled time, waves of pairs times a
  // range's K blocks (0.26 us each at 256 columns) and about 4 us of epilogue, plus the
  // residues written and read (nominal rates), among those whose residues fit
  const int64_t items = (int64_t)g.gm * g.gn * kMod;
  const size_t plane = (size_t)kMod * g.Mr * g.Np;
  double best = 1e300;
  g.gz = 1;
  for (int z = 1; z <= std::min(32, std::max(1, g.kb / 4)); ++z) {
    if (z > 1 && z * plane > kOzResidueCap) break;
    const double waves = (double)((items * z + pairs - 1) / pairs);
    const double t = waves * ((g.kb + z - 1) / z * 1e-9 * g.bn + 4e-6) +
                     z * 2.0 * kMod * (double)g.Mr * g.Nr / 6e12;
    if (t < best) {
      best = t;
      g.gz = z;
    }
  }
  g.kb_per = (g.kb + g.gz - 1) / g.gz;
  g.gz = (g.kb + g.kb_per - 1) / g.kb_per;
  // blocks a row norm: about two waves of 256-thread blocks
  const int rows_a = conjA ? M : (M + 255) / 256;
  g.Sa = std::max(1, std::min({16, (1216 + rows_a - 1) / rows_a, (K + 31) / 32}));
  g.Sb = std::max(1, std::min({16, (1216 + N - 1) / N, (K + 255) / 256}));
  g.bytes_a = oz_align((size_t)kMod * g.Mr * g.seg * 2);
  g.bytes_b = oz_align((size_t)kMod * g.Nr * g.seg * 2);
  g.bytes_r = oz_align(g.gz * plane);
  // norms and exponents: one of a row of A, two of a column
  const size_t pa = conjA ? 2 : 1;
  g.bytes_n = oz_align(((size_t)M * g.Sa * pa + (size_t)N * g.Sb * 2) * 8);
  g.bytes_e = oz_align((M * pa + 2 * (size_t)N) * 4);
  return g;
}

// Pieces of the output, rows by columns, in equal parts of the larger side until
// the result's residues fit, and the operands' over a K of at most 16,384 (long K
// segments keep the MMA pipeline full).
struct ModSplit {
  int pm, pn;
};
inline ModSplit mod_split(bool conjA, int M, int N, int K) {
  const int64_t kreal = std::min<int64_t>(oz_round_up((int64_t)K * (conjA ? 1 : 2), 64), 16384);
  int64_t a = 1, b = 1;
  ModSplit sp{M, N};
  auto part = [](int n, int64_t parts) {
    return (int)std::min<int64_t>(n, oz_round_up((n + parts - 1) / parts, 128));
  };
  for (;;) {
    const ModTiles t = mod_tiles(conjA, sp.pm, sp.pn);
    if ((size_t)(t.Mr + t.Nr) * 2 * kMod * kreal <= kOzOperandCap &&
        (size_t)kMod * t.Mr * t.Np <= kOzResidueCap)
      return sp;
    // the next count of parts that makes them smaller
    if (t.Mr >= t.Nr) {
      const int was = sp.pm;
      while (sp.pm == was) sp.pm = part(M, ++a);
    } else {
      const int was = sp.pn;
      while (sp.pn == was) sp.pn = part(N, ++b);
    }
  }
}

// An upper bound of the workspace of any product of at most these sizes.
inline size_t mod_bound(bool conjA, int M, int N, int K) {
  const int64_t kreal = oz_round_up((int64_t)K * (conjA ? 1 : 2), 64);
  const ModTiles t = mod_tiles(conjA, M, N);
  const size_t a = (size_t)(t.Mr + t.Nr) * 2 * kMod;  // bytes a real K
  const size_t operands = a > kOzOperandCap / kreal ? kOzOperandCap : a * kreal;
  // (Np of fewer columns is at most this)
  const size_t plane = (size_t)kMod * t.Mr * (size_t)std::min<int64_t>(256 * (int64_t)t.gn, t.Nr + 32 * t.gn);
  const size_t ranges = (size_t)std::min<int64_t>(32, std::max<int64_t>(1, kreal / 256));
  const size_t residues = std::min(kOzResidueCap, plane > kOzResidueCap ? kOzResidueCap : plane * ranges);
  // rows of a piece: their operand residues over 64 of K fit
  const size_t rows = std::min<size_t>((size_t)M + N, kOzOperandCap / (2 * kMod * 64) + 256);
  return operands + residues + rows * 2 * (16 * 8 + 4) + 5 * 256;
}

}  // namespace pwh

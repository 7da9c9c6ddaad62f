"""The fused double-float operations of the FP64 FFT passes (csrc/fft_df.cuh) and
the transforms built from them (csrc/fft_spec_impl.cuh), on the host.

Operations, against exact rationals, cancelling operands included.  The sum: 2^-44
of the result, as operator+ (test_df_arith.py), its low part normalised to 2^-48 of
the operands.  a b + c d and z + a b + c d:
each product's small terms are at most 2 2^-24 of it and pass through at most eight
FP32 roundings, 2^-24 each, besides the dropped product of low parts: 2^-44 of the
sum of the terms' magnitudes.

Transforms: the rms error of one forward transform of random data at every compiled
edge is no larger than with the composed operations of df.cuh in four-step form
(the arithmetic before the fused operations), 1% for the sampling (3 standard
deviations of the ratio over 300 transforms)."""
import random
import subprocess
from fractions import Fraction

import pytest

from tests.test_df_arith import CSRC, _nvcc, bits, exact, f32, pair, rnd32

PROG = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>
#include "fft_df.cuh"
#include "fft_spec_impl.cuh"
using namespace pwh;
static float f_of(uint32_t u) { float f; std::memcpy(&f, &u, 4); return f; }
static uint32_t u_of(float f) { uint32_t u; std::memcpy(&u, &f, 4); return u; }
typedef long double LD;

template <class T, int N> void transform(cx<T>* x, const cx<T>* tw) {
  using F = Fac<T, N>;
  for (int n2 = 0; n2 < F::N2; ++n2) {
    cx<T> v[F::N1];
    for (int i = 0; i < F::N1; ++i) v[i] = x[F::idx_a(i, n2)];
    dft_reg<T, F::N1, false, N>(v, tw);
    if constexpr (!F::pfa)
      for (int k = 1; k < F::N1; ++k) v[k] = mul<T>(v[k], signed_tw<T, false>(tw[n2 * k]));
    for (int i = 0; i < F::N1; ++i) x[F::idx_a(i, n2)] = v[i];
  }
  std::vector<cx<T>> o(N);
  for (int k1 = 0; k1 < F::N1; ++k1) {
    cx<T> w[F::N2];
    for (int i = 0; i < F::N2; ++i) w[i] = x[F::idx_a(k1, i)];
    dft_reg<T, F::N2, false, N>(w, tw);
    for (int i = 0; i < F::N2; ++i) o[F::idx_b(k1, i)] = w[i];
  }
  for (int i = 0; i < N; ++i) x[i] = o[i];
}
template <class T, int N> double rms() {
  std::mt19937_64 g(N);
  std::normal_distribution<double> d;
  std::vector<cx<T>> tw(N);
  std::vector<LD> c(N), s(N);
  for (int i = 0; i < N; ++i) {
    c[i] = cosl(2 * acosl(-1.0L) * i / N);
    s[i] = sinl(2 * acosl(-1.0L) * i / N);
    tw[i].x = T(df((double)c[i]));
    tw[i].y = T(df((double)s[i]));
  }
  double e2 = 0, r2 = 0;
  for (int r = 0; r < 300; ++r) {
    std::vector<cx<T>> x(N);
    std::vector<LD> a(N), b(N);
    for (int i = 0; i < N; ++i) {
      const df p(d(g)), q(d(g));
      x[i].x = T(p);
      x[i].y = T(q);
      a[i] = (LD)p.hi + p.lo;
      b[i] = (LD)q.hi + q.lo;
    }
    transform<T, N>(x.data(), tw.data());
    for (int k = 0; k < N; ++k) {
      LD u = 0, v = 0;
      for (int n = 0; n < N; ++n) {
        const int t = n * k % N;
        u += a[n] * c[t] + b[n] * s[t];
        v += b[n] * c[t] - a[n] * s[t];
      }
      const LD du = (LD)x[k].x.hi + x[k].x.lo - u, dv = (LD)x[k].y.hi + x[k].y.lo - v;
      e2 += (double)(du * du + dv * dv);
      r2 += (double)(u * u + v * v);
    }
  }
  return std::sqrt(e2 / r2);
}
int main(int argc, char**) {
  if (argc > 1) {
#define ROW(n) std::printf("%d %.6e %.6e\n", n, rms<dfa, n>(), rms<DfPass<n>, n>());
    PWH_SPEC_SIZES(ROW)
    return 0;
  }
  char op[8];
  unsigned u[10];
  while (std::scanf("%7s", op) == 1) {
    df x[5];
    for (int i = 0; i < 5; ++i) {
      if (std::scanf("%x %x", u, u + 1) != 2) return 1;
      x[i] = df(f_of(u[0]), f_of(u[1]));
    }
    const df r = op[0] == 's' ? df_sum(x[0], x[1])
                 : op[0] == '2' ? df_dot2(x[0], x[1], x[2], x[3]) : df_dot3(x[4], x[0], x[1], x[2], x[3]);
    std::printf("%08x %08x\n", u_of(r.hi), u_of(r.lo));
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    nv = _nvcc()
    if nv is None:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("dft")
    src = d / "dft_host.cu"
    src.write_text(PROG)
    out = d / "dft_host"
    subprocess.run([nv, "-std=c++17", "--expt-relaxed-constexpr", "-O2", "-w", "-Xcompiler",
                    "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(out)],
                   check=True, capture_output=True, timeout=600)
    return str(out)


def near(rng, x, rel):
    """A normalised pair close to -x: the high parts cancel up to rel."""
    hi = rnd32(-x[0] * (1 + rng.uniform(-1, 1) * rel))
    return hi, rnd32(hi * rng.uniform(-1, 1) * 2.0 ** -25)


@pytest.mark.parametrize("op", ["s", "2", "3"])
def test_fused_operations_within_bound(exe, op):
    rng = random.Random(ord(op))
    cases = []
    for i in range(4000):
        a, b, c, d, z = (pair(rng) for _ in range(5))
        k = i % 4
        if op == "s" and k:
            b = near(rng, a, (0.0, 2.0 ** -22, 2.0 ** -10)[k - 1])
        elif op == "2" and k:
            c, d = near(rng, a, (0.0, 2.0 ** -22, 2.0 ** -10)[k - 1]), b
        elif op == "3" and k:
            z = near(rng, (rnd32(a[0] * b[0] + c[0] * d[0]), 0.0), (0.0, 2.0 ** -22, 2.0 ** -10)[k - 1])
        cases.append((a, b, c, d, z))
    lines = [op + "".join(f" {bits(p[0]):08x} {bits(p[1]):08x}" for p in q) for q in cases]
    p = subprocess.run([exe], input="\n".join(lines) + "\n", capture_output=True, text=True, check=True,
                       timeout=60)
    out = [tuple(f32(int(t, 16)) for t in l.split()) for l in p.stdout.strip().splitlines()]
    assert len(out) == len(cases)
    for q, (hi, lo) in zip(cases, out):
        a, b, c, d, z = (exact(*v) for v in q)
        terms = {"s": (a, b), "2": (a * b, c * d), "3": (z, a * b, c * d)}[op]
        ref = sum(terms)
        scale = abs(ref) if op == "s" else sum(abs(t) for t in terms)
        assert abs(exact(hi, lo) - ref) <= Fraction(1, 2 ** 44) * scale, (op, q, hi, lo)
        slack = max(abs(a), abs(b)) / 2 ** 48 if op == "s" else 0
        assert abs(exact(lo)) <= abs(exact(hi)) * Fraction(2.0 ** -23.99) + slack


def test_transforms_no_less_accurate_than_composed(exe):
    p = subprocess.run([exe, "t"], capture_output=True, text=True, check=True, timeout=600)
    rows = [l.split() for l in p.stdout.strip().splitlines()]
    assert len(rows) == 12
    worse = {n: float(f) / float(c) for n, c, f in rows if float(f) > 1.01 * float(c)}
    assert not worse

"""The end of the CTA pair's ring (csrc/pair_ring.cuh) in a model of its barriers, on the
host: a fill's copies complete on CTA 0's barrier of the slot, which CTA 0 arms for both
CTAs' bytes when it fills the slot itself.  Producers, copies and the consumer proceed in
random order and stop at random, as after a time-out; whatever the two counts are, the
end must arm only the current phase of a barrier, and wait for every slot that has a
copy in flight."""
import shutil
import subprocess

import pytest

from tests.test_df_arith import CSRC

PROG = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "pair_ring.cuh"
using pwh::PairDrain;
struct Copy { int cta, fill; };
int main() {
  std::mt19937 g(3);
  auto rnd = [&](int n) { return (int)(g() % (unsigned)n); };
  int apart = 0;
  for (int run = 0; run < 200000; ++run) {
    const int S = 2 + rnd(5), total = rnd(4 * S + 1);
    int fills[2] = {0, 0}, used = 0;       // slots filled by each CTA, consumed
    int phase[8] = {}, armed[8] = {}, tx[8] = {};  // CTA 0's barriers: phases done, pending arrival made, bytes
    std::vector<Copy> flight;
    bool stopped[2] = {false, false};
    auto settle = [&](int s) {
      if (armed[s] && tx[s] == 0) { armed[s] = 0; ++phase[s]; }
    };
    auto land = [&](size_t i) {
      const int s = flight[i].fill % S;
      --tx[s];
      flight.erase(flight.begin() + i);
      settle(s);
    };
    for (int step = 0; step < 6 * total; ++step) {
      const int what = rnd(5);
      if (what < 2) {
        const int r = what;
        if (rnd(12) == 0) stopped[r] = true;
        // a slot is free once its previous fill was consumed
        if (stopped[r] || fills[r] >= total || fills[r] - S >= used) continue;
        const int s = fills[r] % S;
        if (r == 0) { armed[s] = 1; tx[s] += 2; }
        flight.push_back({r, fills[r]++});
      } else if (what == 2) {
        if (used < fills[0] && phase[used % S] > used / S) ++used;
      } else if (!flight.empty()) {
        land(rnd((int)flight.size()));
      }
    }
    const PairDrain d = pwh::pair_drain(fills[0], fills[1], S);
    apart += fills[0] != fills[1];
    for (int j = d.arm0; j < d.arm1; ++j) {
      if (phase[j % S] != j / S || armed[j % S]) return std::printf("run %d: fill %d armed early\n", run, j), 1;
      armed[j % S] = 1;
      tx[j % S] += 1;
      settle(j % S);
    }
    for (const Copy& c : flight)
      if (c.fill < d.wait0 || c.fill >= d.wait1) return std::printf("run %d: fill %d not waited for\n", run, c.fill), 1;
    while (!flight.empty()) land(rnd((int)flight.size()));
    for (int j = d.wait0; j < d.wait1; ++j)
      // the wait of a fill that both made, or CTA 1 alone, ends
      if (j < fills[1] && phase[j % S] != j / S + 1) return std::printf("run %d: fill %d not complete\n", run, j), 1;
  }
  std::printf("%d\n", apart);
  return 0;
}
"""


def test_every_copy_is_waited_for(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    src = tmp_path / "ring.cpp"
    src.write_text(PROG)
    out = tmp_path / "ring"
    subprocess.run([gxx, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(out)], check=True, timeout=120)
    r = subprocess.run([str(out)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 1000          # runs whose producers stopped apart

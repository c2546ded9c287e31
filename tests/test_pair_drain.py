"""lm_pair_drain, the end of a CTA pair's producers after one of them has given up (a bounded wait that ran out), against
a model of CTA 0's full barriers on the host: for every pair of slab counts that the two can have, and copies that land
in any order, the drain ends with every copy of both CTAs landed."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MODEL = r"""
#include <cstdio>
#include <random>
#include <vector>
#include "lm_head.cuh"

// a full barrier: one arrival a phase, and the bytes expected less those landed
struct Bar {
  int pending = 1, phase = 0;
  long tx = 0;
  void turn() {
    if (pending == 0 && tx == 0) { pending = 1; ++phase; }
  }
  void arrive_expect(long b) { tx += b; --pending; turn(); }
  void landed(long b) { tx -= b; turn(); }
};
constexpr long SHARE = 100;
struct Ring {
  std::vector<Bar> bar;
  std::vector<uint32_t> flying;  // stages of the copies on their way
  std::mt19937 rng;
  void land_one() {
    const size_t i = rng() % flying.size();
    const uint32_t w = flying[i];
    flying.erase(flying.begin() + i);
    bar[w].landed(SHARE / 2);  // W and H of one CTA's share come one by one
  }
  void ask(uint32_t w, bool first) {
    if (first) bar[w].arrive_expect(2 * SHARE);
    flying.push_back(w);
    flying.push_back(w);
  }
  void expect_one(uint32_t w) { bar[w].arrive_expect(SHARE); }
  void missing_one(uint32_t w) { bar[w].landed(SHARE); }
  bool wait(uint32_t w, uint32_t parity) {  // true once the phase of that parity is over
    while ((uint32_t)(bar[w].phase & 1) == parity) {
      if (flying.empty()) return false;
      land_one();
    }
    return true;
  }
};

int main() {
  int runs = 0;
  for (uint32_t stages = 2; stages <= 12; ++stages)
    for (uint32_t used = 0; used <= 2 * stages + 1; ++used)  // slabs consumed before the MMAs stopped
      for (uint32_t n0 = used; n0 <= used + stages; ++n0)
        for (uint32_t n1 = used; n1 <= used + stages; ++n1) {
          Ring r;
          r.bar.resize(stages);
          r.rng.seed(runs);
          for (uint32_t j = 0; j < used; ++j) {
            r.ask(j % stages, true);
            r.ask(j % stages, false);
            while (!r.flying.empty()) r.land_one();
          }
          uint32_t a = used, b = used;
          while (a < n0 || b < n1) {  // the two CTAs in any order
            if (b == n1 || (a < n0 && (r.rng() & 1))) r.ask(a++ % stages, true);
            else r.ask(b++ % stages, false);
            if (!r.flying.empty() && r.rng() % 3 == 0) r.land_one();
          }
          const bool done = pced::lm_pair_drain(n0, n1, stages, r);
          if (!done || !r.flying.empty()) {
            printf("stages %u used %u n0 %u n1 %u: done %d, %zu copies flying\n", stages, used, n0, n1, done,
                   r.flying.size());
            return 1;
          }
          ++runs;
        }
  printf("%d\n", runs);
  return 0;
}
"""


def test_drain_ends_with_every_copy_landed(tmp_path):
    src, exe = tmp_path / "drain.cu", tmp_path / "drain"
    src.write_text(MODEL)
    subprocess.check_call(["nvcc", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                           "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_2601_08670_gb300", "csrc"), "-o", str(exe), str(src)])
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0, res.stdout
    assert int(res.stdout) > 10000

"""The sums of the dynamic contrast strength (three fp32 numbers, csrc/sum3.cuh), compiled for the host, against exact
sums: no further off than an fp64 accumulator may be, n 2^-53 of the terms' magnitudes for n terms."""
import os
import random
import subprocess
from fractions import Fraction

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_08670_gb300", "csrc")

MAIN = r"""
#define __host__
#define __device__
#define __forceinline__ inline
#include "sum3.cuh"
#include <cstdio>
#include <vector>
// lines "lanes n" and n terms: lane i takes terms i, i + lanes, ..., then the lanes in a tree
int main() {
  int lanes, n;
  while (scanf("%d %d", &lanes, &n) == 2) {
    std::vector<float> t(n);
    for (float& x : t) scanf("%a", &x);
    std::vector<pced::Sum3> p(lanes, pced::Sum3{0.f, 0.f, 0.f});
    for (int i = 0; i < lanes; ++i)
      for (int j = i, k = 1; j < n; j += lanes, ++k) {
        pced::sum3_add(p[i], t[j]);
        if (k % pced::SUM3_RUN == 0) pced::sum3_settle(p[i]);
      }
    for (int o = lanes / 2; o > 0; o /= 2)
      for (int i = 0; i < o; ++i) p[i] = pced::sum3_merge(p[i], p[i + o]);
    printf("%a\n", pced::sum3_value(p[0]));
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def sums(tmp_path_factory):
    d = tmp_path_factory.mktemp("sum3")
    (d / "main.cpp").write_text(MAIN)
    subprocess.check_call(["g++", "-O2", "-ffp-contract=off", "-I", CSRC, "-o", str(d / "main"), str(d / "main.cpp")])

    def run(lanes, terms):
        text = f"{lanes} {len(terms)}\n" + "\n".join(float(t).hex() if abs(t) < 1e300 else str(t) for t in terms) + "\n"
        out = subprocess.run([str(d / "main")], input=text, capture_output=True, text=True, check=True).stdout
        return float.fromhex(out.strip())
    return run


def _f32(x):
    import numpy as np
    return float(np.float32(x))


def _cases():
    rng = random.Random(1)
    # terms that a pair of fp32 numbers drops one by one: under half an ulp of its low part
    yield 1, [1.0, 2.0 ** -24 * 1.5] + [2.0 ** -49 * 1.9] * 123
    yield 32, [1.0] * 32 + [2.0 ** -24 * 1.5] * 32 + [2.0 ** -49 * 1.9] * 4000
    yield 1, ([1.0] + [2.0 ** -24 * 1.5] * 30 + [2.0 ** -48 * 1.1] * 96) * 100
    yield 1, [2.0 ** -49 * 1.9] * 123 + [2.0 ** -24 * 1.5, 1.0]
    # probabilities' terms over many orders of magnitude; signs as rounding leaves them
    for lanes, n in ((1, 5), (1, 20000), (32, 1000), (32, 16032), (1024, 128256)):
        yield lanes, [_f32(rng.choice([1, 1, 1, -1e-3]) * 10.0 ** rng.uniform(-30, 0)) for _ in range(n)]
    yield 4, [_f32(10.0 ** rng.uniform(-44, -36)) for _ in range(500)]  # down into the subnormal numbers


@pytest.mark.parametrize("lanes,terms", list(_cases()), ids=lambda x: None if isinstance(x, list) else str(x))
def test_no_less_exact_than_fp64(sums, lanes, terms):
    exact = sum(Fraction(t) for t in terms)
    bound = len(terms) * Fraction(1, 2 ** 53) * sum(abs(Fraction(t)) for t in terms)
    assert abs(Fraction(sums(lanes, terms)) - exact) <= bound


@pytest.mark.parametrize("terms", [[1.0, float("inf"), 2.0, 3.0, 4.0], [3e38] * 9])
def test_infinite_sums_stay_infinite(sums, terms):
    assert sums(2, terms) == float("inf")


def test_nan_terms_give_nan(sums):
    assert sums(2, [1.0, float("nan"), 2.0]) != sums(2, [1.0, float("nan"), 2.0])

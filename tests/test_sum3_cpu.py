"""The three-word FP32 sum (csrc/sum3.cuh), compiled for the host, against exact
rational sums. Bounds: the words together are rounded once to FP64 (2^-53 of the
sum); what the third word rounds off is at most (number of summands) 2^-24 of its
own size, itself below (number of summands) 2^-48 of the sum of magnitudes."""
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include <cmath>
#include <cstdio>
#define __device__
#define __forceinline__ inline
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmul_rn(float a, float b) { return a * b; }
static float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
#include "sum3.cuh"
int main() {
  int square, n;
  while (std::scanf("%d %d", &square, &n) == 2) {
    Sum3 s;
    for (int i = 0; i < n; ++i) {
      float v;
      if (std::scanf("%a", &v) != 1) return 1;
      if (square) s.add_square(v); else s.add(v);
    }
    std::printf("%a\n", s.value());
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("sum3")
    (d / "cuda_runtime.h").write_text("#pragma once\n")
    (d / "main.cpp").write_text(MAIN)
    csrc = os.path.join(ROOT, "paper_2303_02346_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", f"-I{d}", f"-I{csrc}", str(d / "main.cpp"),
                    "-o", str(d / "main")], check=True)
    return str(d / "main")


@pytest.mark.parametrize("square", [0, 1])
@pytest.mark.parametrize("kind", ["positive", "mixed", "cancelling", "spread", "equal"])
def test_against_exact_sums(program, kind, square):
    rng = np.random.default_rng(5)
    runs = []
    for n in (1, 2, 7, 16, 24, 64):
        for _ in range(20):
            v = rng.uniform(0.1, 1, n) if kind == "positive" else rng.normal(size=n)
            if kind == "spread":
                v = v * 10.0 ** rng.uniform(-6, 6, n)
            if kind == "equal":
                v = np.full(n, v[0])
            v = v.astype(np.float32)
            if kind == "cancelling":
                v = np.concatenate([v, -v * np.float32(1 + 2 ** -20)]).astype(np.float32)
            runs.append(v)
    text = "".join(f"{square} {len(v)} " + " ".join(float(t).hex() for t in v) + "\n" for v in runs)
    out = subprocess.run([program], input=text, capture_output=True, text=True, check=True).stdout.split()
    assert len(out) == len(runs)
    for v, got in zip(runs, out):
        terms = [Fraction(float(t)) ** (2 if square else 1) for t in v]
        exact, size, n = sum(terms), sum(abs(t) for t in terms), len(v) * (2 if square else 1)
        bound = abs(exact) * Fraction(1, 2 ** 53) + size * n * n * Fraction(1, 2 ** 72)
        assert abs(Fraction(float.fromhex(got)) - exact) <= bound

"""CPU test of the three-float sums (csrc/tri.h) that stand for FP64 in the inner iteration on
FP32 vectors: dot products, quotients and products of scalars, and the vector updates, each
against exact rationals, with the error FP64 arithmetic may have as the bound."""

import math
import os
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1008_1700_gb300", "csrc")
MAIN = r"""
#include <cstdio>
#include "tri.h"
using namespace ddps;
static void out(Tri t) { std::printf("%a %a %a\n", t.h, t.m, t.l); }
int main() {
  char op[8];
  int n;
  while (std::scanf("%7s %d", op, &n) == 2) {
    float v[8192];
    for (int i = 0; i < n; ++i) std::scanf("%f", v + i);
    const Tri a{v[0], v[1], v[2]}, b{v[3], v[4], v[5]};
    if (op[0] == 'd') {  // dot of the halves: eight strided sums, then a tree, as over lanes
      Tri s[8] = {};
      for (int i = 0; i < n / 2; ++i) s[i % 8] = sum(s[i % 8], mul(v[i], v[n / 2 + i]));
      for (int o = 4; o; o /= 2)
        for (int i = 0; i < o; ++i) s[i] = sum(s[i], s[i + o]);
      out(settle(s[0]));
    } else if (op[0] == 'q') {
      out(quot(a, b));
    } else if (op[0] == 'm') {
      out(mul(a, b));
    } else if (op[0] == 'l') {
      std::printf("%a %a\n", lin(v[6], a, v[7]), lin(v[6], a, v[7], b, v[8]));
    } else {
      std::printf("%d %d\n", (int)less(a, b), (int)at_most(a, b));
    }
  }
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("tri")
    src, exe = d / "main.cpp", d / "main"
    src.write_text(MAIN)
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)

    def call(cases):
        text = "\n".join(f"{op} {len(v)} " + " ".join(float(np.float32(x)).hex() for x in v)
                         for op, v in cases)
        r = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True)
        return [line.split() for line in r.stdout.splitlines()]
    return call


def _tri(rng, lo=-8, hi=8):
    x = math.ldexp(rng.uniform(1.0, 2.0), int(rng.integers(lo, hi))) * rng.choice([-1, 1])
    h = np.float32(x)
    m = np.float32(x - float(h))
    return [h, m, np.float32(rng.uniform(-1, 1) * 2.0 ** -25 * float(m))]


def _value(words):
    return sum(Fr(float.fromhex(w)) for w in words)


@pytest.mark.parametrize("n", [1, 7, 128, 1001])
@pytest.mark.parametrize("spread", [0, 12])
@pytest.mark.parametrize("scale", [20, -37])  # ||g||, and a residual 10^-17 of it
def test_dot_products(run, n, spread, scale):
    rng = np.random.default_rng([n, spread, scale + 64])
    v = [np.ldexp(rng.uniform(-1, 1, 2 * n), rng.integers(-spread, spread + 1, 2 * n) + scale)
         .astype(np.float32) for _ in range(20)]
    v += [np.concatenate([np.sort(w[:n]), w[n:] * np.sign(rng.uniform(-1, 1, n))]) for w in v]  # cancelling
    for w, got in zip(v, run([("d", w) for w in v])):
        p = [Fr(float(x)) * Fr(float(y)) for x, y in zip(w[:n], w[n:])]
        # FP64: one rounding of 2^-53 a term, of partial sums up to the sum of magnitudes
        assert abs(_value(got) - sum(p)) <= Fr(2) ** -53 * sum(abs(x) for x in p)


def test_scalars(run):
    rng = np.random.default_rng(1)
    cases = [_tri(rng) + _tri(rng) for _ in range(400)]
    for c, q, m in zip(cases, run([("q", c) for c in cases]), run([("m", c) for c in cases])):
        a, b = (sum(Fr(float(x)) for x in c[o:o + 3]) for o in (0, 3))
        assert abs(_value(q) - a / b) <= Fr(2) ** -53 * abs(a / b)
        assert abs(_value(m) - a * b) <= Fr(2) ** -53 * abs(a * b)


def test_updates(run):
    rng = np.random.default_rng(2)
    cases = []
    for i in range(600):
        a, b = _tri(rng), _tri(rng)
        x, y = (np.float32(rng.uniform(-4, 4)) for _ in range(2))
        r = np.float32(rng.uniform(-4, 4))
        if i % 2:  # cancelling
            r = np.float32(-(float(a[0]) * float(x) + (float(b[0]) * float(y) if i % 4 == 1 else 0.0)))
        cases.append(a + b + [r, x, y])
    for c, (l1, l2) in zip(cases, run([("l", c) for c in cases])):
        a, b = (sum(Fr(float(x)) for x in c[o:o + 3]) for o in (0, 3))
        r, x, y = (Fr(float(v)) for v in c[6:])
        for got, terms in ((l1, [r, a * x]), (l2, [r, a * x, b * y])):
            # FP64: a rounding of 2^-53 of the terms each, then the one to a float
            exact = sum(terms)
            bound = Fr(2) ** -24 * abs(exact) + 4 * Fr(2) ** -53 * sum(abs(t) for t in terms)
            assert abs(Fr(float.fromhex(got)) - exact) <= bound


def test_comparisons(run):
    one, below = [1.0, 0.0, 0.0], [1.0, 0.0, -2.0 ** -60]
    nan = [math.nan, 0.0, 0.0]
    got = run([("c", v) for v in (one + one, below + one, one + below, nan + one, one + nan)])
    assert got == [["0", "1"], ["1", "1"], ["0", "0"], ["0", "0"], ["0", "0"]]

"""Host checks of the double-float arithmetic of the streaming tier, compiled from the shipped header
(``mq_df.cuh``) behind host definitions of the rounding intrinsics: the integer split of a double
keeps 48 bits (and keeps zeros, signs and non-finite values), and sums, differences and products
stay within the bounds of the published algorithms (a few units of 2^-48)."""
import os
import random
import shutil
import struct
import subprocess
from fractions import Fraction

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <algorithm>
#define __device__
#define __forceinline__ inline
using std::max; using std::min;
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
static inline float __uint_as_float(unsigned u) { float f; std::memcpy(&f, &u, 4); return f; }
static inline long long __double_as_longlong(double d) { long long b; std::memcpy(&b, &d, 8); return b; }
template <typename T> static inline T __shfl_xor_sync(unsigned, T v, int) { return v; }
"""
MAIN = r"""
int main() {
  char op; unsigned long long a, b;
  while (std::scanf(" %c %llx %llx", &op, &a, &b) == 3) {
    double x, y; std::memcpy(&x, &a, 8); std::memcpy(&y, &b, 8);
    using namespace mq::dev;
    const df p = df_split(x), q = df_split(y);
    df r = p;
    if (op == '+') r = df_add(p, q);
    if (op == '-') r = df_sub(p, q);
    if (op == '*') r = df_mul(p, q);
    std::printf("%a %a\n", (double)r.h, (double)r.l);
  }
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("df")
    body = open(os.path.join(ROOT, "paper_2103_03407_gb300", "csrc", "mq_df.cuh")).read()
    body = body.replace("#pragma once", "").replace("#include <cuda_runtime.h>", "")
    (d / "t.cpp").write_text(SHIM + body + MAIN)
    subprocess.run([cxx, "-std=c++17", "-O1", "-ffp-contract=off", "-o", str(d / "t"), str(d / "t.cpp")], check=True)

    def call(rows):
        bits = lambda v: struct.unpack("<Q", struct.pack("<d", v))[0]  # noqa: E731
        text = "".join("%s %x %x\n" % (o, bits(x), bits(y)) for o, x, y in rows)
        out = subprocess.run([str(d / "t")], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(float.fromhex(v) if "n" not in v else float(v) for v in ln.split()) for ln in out.splitlines()]

    return call


def test_split_keeps_48_bits(run):
    rng = random.Random(1)
    vals = [rng.choice([-1, 1]) * (1 + rng.random()) * 2.0 ** rng.randint(-70, 100) for _ in range(4000)]
    vals += [1.0, -1.0, 1 + 2.0 ** -52, 2 - 2.0 ** -52, 1 + 2.0 ** -24, 1 - 2.0 ** -53, 2.0 ** -73]
    for v, (h, l) in zip(vals, run([("s", v, 0.0) for v in vals])):
        assert abs(Fraction(h) + Fraction(l) - Fraction(v)) <= abs(Fraction(v)) * Fraction(1, 2 ** 47), v
        assert abs(l) <= abs(h) * 2.0 ** -23
    inf = float("inf")
    (z, zl), (p, _), (m, _), (q, _) = run([("s", v, 0.0) for v in (0.0, inf, -inf, float("nan"))])
    assert z == 0.0 and zl == 0.0 and p == inf and m == -inf and q != q


@pytest.mark.parametrize("op", ["+", "-", "*"])
def test_operations_within_published_bounds(run, op):
    # x and y enter with 48 bits each (relative 2^-47 of each operand); a sum adds at most 2 units of
    # 2^-48 of the operands (cancellation), a product of two positive factors 8 units of itself
    rng = random.Random(2)
    rows = []
    for _ in range(4000):
        x = rng.choice([-1, 1]) * (1 + rng.random()) * 2.0 ** rng.randint(-20, 20)
        y = x * (1 + rng.random() * 2.0 ** rng.randint(-40, 4)) if rng.random() < 0.5 else rng.uniform(-1, 1) * x
        rows.append((op, x, y))
    for (_, x, y), (h, l) in zip(rows, run(rows)):
        X, Y, got = Fraction(x), Fraction(y), Fraction(h) + Fraction(l)
        if op == "*":
            ref, tol = X * Y, abs(X * Y) * 16
        else:
            ref, tol = (X + Y if op == "+" else X - Y), (abs(X) + abs(Y)) * 8
        assert abs(got - ref) <= tol / 2 ** 48, (x, y)

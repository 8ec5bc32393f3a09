"""The integer fold of the tensor-core coefficient kernels over their whole domain |y| <= 1, compiled for the host from the
shipped source: at the largest group sums that this domain allows, (g + 2) 16 T 2^14, every group converts
exactly (short contractions: by the form small_groups chooses) and the fold is the exact sum modulo 2^64."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#define __device__
#define __forceinline__ inline
static inline int __float2int_rn(float f) { return (int)std::nearbyint(f); }
static inline float __uint_as_float(uint32_t u) { float f; std::memcpy(&f, &u, 4); return f; }
static inline int __float_as_int(float f) { int i; std::memcpy(&i, &f, 4); return i; }
static inline uint32_t bits(int v) { float f = (float)v; uint32_t u; std::memcpy(&u, &f, 4); return u; }
"""
MAIN = r"""
template <int SMALL>
static long long resident(const int* s, int fs, long long w) {
  return fold_fixed(group_sum_if<(SMALL > 0)>(bits(s[0])) * 256 + group_sum_if<(SMALL > 1)>(bits(s[1])),
                    group_sum_if<(SMALL > 2)>(bits(s[2])) * 256 + group_sum_if<(SMALL > 3)>(bits(s[3])),
                    group_sum_if<(SMALL > 4)>(bits(s[4])), group_sum(bits(s[5])), group_sum(bits(s[6])), fs, w);
}
int main() {
  int T, fs, s[7];
  long long w;
  while (std::scanf("%d %d %lld %d %d %d %d %d %d %d", &T, &fs, &w, s, s + 1, s + 2, s + 3, s + 4, s + 5, s + 6) == 10) {
    long long r;
    if (T > 5)
      r = fold_fixed(group_sum(bits(s[0])) * 256 + group_sum(bits(s[1])),
                     (long long)group_sum(bits(s[2])) * 256 + group_sum(bits(s[3])), group_sum(bits(s[4])),
                     group_sum(bits(s[5])), group_sum(bits(s[6])), fs, w);
    else
      r = T <= 2 ? resident<small_groups(2)>(s, fs, w) : T == 3 ? resident<small_groups(3)>(s, fs, w)
          : T == 4 ? resident<small_groups(4)>(s, fs, w) : resident<small_groups(5)>(s, fs, w);
    std::printf("%llu\n", (unsigned long long)r);
  }
}
"""


@pytest.fixture(scope="module")
def fold(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    src = open(os.path.join(ROOT, "paper_2103_03407_gb300", "csrc", "mq_tc.cu")).read()
    i = src.index("__device__ __forceinline__ int group_sum(uint32_t r)")
    body = src[i:src.index("// start of output row b", i)]
    d = tmp_path_factory.mktemp("fold")
    (d / "t.cpp").write_text(SHIM + body + MAIN)
    subprocess.run([cxx, "-std=c++17", "-O1", "-fwrapv", "-o", str(d / "t"), str(d / "t.cpp")], check=True)

    def run(rows):
        text = "".join(" ".join(map(str, r)) + "\n" for r in rows)
        out = subprocess.run([str(d / "t")], input=text, capture_output=True, text=True, check=True).stdout
        return [int(v) for v in out.split()]

    return run


def test_fold_at_the_largest_group_sums(fold):
    rows = []
    for T in (1, 2, 3, 4, 5, 8):
        top = [(g + 2) * 16 * T << 14 for g in range(7)]
        for fs in range(1, 9):
            for m in range(128):  # every choice of signs, and one off the largest values
                s = [(-v if m >> g & 1 else v) for g, v in enumerate(top)]
                rows.append([T, fs, 12345, *s])
                rows.append([T, fs, -(1 << 62), *(v - (1 if v > 0 else -1) for v in s)])
    for (T, fs, w, *s), got in zip(rows, fold(rows)):
        ref = w + sum(v * 2 ** (8 * (6 - g)) >> fs for g, v in enumerate(s[:6])) + (s[6] >> fs)
        assert got == ref % 2 ** 64, (T, fs, s)


def test_the_launch_uses_these_bounds():
    src = open(os.path.join(ROOT, "paper_2103_03407_gb300", "csrc", "mq_tc.cu")).read()
    assert set(re.findall(r"k_coef_res<([^>]*)>", src)) == {"small_groups(%d)" % t for t in (2, 3, 4, 5)}

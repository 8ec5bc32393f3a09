// Double-float arithmetic: a value as the unevaluated sum of two FP32 numbers (about 48 bits).
//
// GB300 issues FP64 at 1/64 of its FP32 rate (one warp instruction per SM and 16 clocks), so a
// double-float sum or product (6 to 11 FP32 instructions, four warp instructions per SM and clock)
// takes a fifth of the time of the FP64 instruction it replaces.  The error-free transformations
// are Knuth's two-sum, Dekker's fast two-sum and the fused-multiply-add product (Dekker 1971;
// Joldes, Muller and Popescu 2017, "Tight and rigorous error bounds for basic building blocks of
// double-word arithmetic").  Every operation is written with the rounding intrinsics, which the
// compiler neither contracts nor reorders.
#pragma once

#include <cuda_runtime.h>

namespace mq {
namespace dev {

struct df {
  float h, l;
};

// a + b = s + e exactly (two-sum)
__device__ __forceinline__ df two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
// a - b = s + e exactly
__device__ __forceinline__ df two_diff(float a, float b) {
  const float s = __fsub_rn(a, b), bb = __fsub_rn(s, a);
  return {s, __fsub_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fadd_rn(b, bb))};
}
// h + l renormalised (|l| <= |h|, or h = 0)
__device__ __forceinline__ df fast_two_sum(float h, float l) {
  const float s = __fadd_rn(h, l);
  return {s, __fsub_rn(l, __fsub_rn(s, h))};
}
// x + y
__device__ __forceinline__ df df_add(df x, df y) {
  const df s = two_sum(x.h, y.h);
  return fast_two_sum(s.h, __fadd_rn(s.l, __fadd_rn(x.l, y.l)));
}
// x - y
__device__ __forceinline__ df df_sub(df x, df y) {
  const df s = two_diff(x.h, y.h);
  return fast_two_sum(s.h, __fadd_rn(s.l, __fsub_rn(x.l, y.l)));
}
// x y, not renormalised: |l| is a few units of h's last place
__device__ __forceinline__ df df_mul(df x, df y) {
  const float p = __fmul_rn(x.h, y.h);
  return {p, __fmaf_rn(x.h, y.l, __fmaf_rn(x.l, y.h, __fmaf_rn(x.h, y.h, -p)))};
}
// x y for a plain FP32 y, not renormalised
__device__ __forceinline__ df df_mul(df x, float y) {
  const float p = __fmul_rn(x.h, y);
  return {p, __fmaf_rn(x.l, y, __fmaf_rn(x.h, y, -p))};
}
// acc += x (x need not be normalised; the sum is left unnormalised: acc.l collects the errors)
__device__ __forceinline__ void df_acc(df& acc, df x) {
  const df s = two_sum(acc.h, x.h);
  acc.h = s.h;
  acc.l = __fadd_rn(acc.l, __fadd_rn(s.l, x.l));
}
__device__ __forceinline__ df df_neg(df x) { return {-x.h, -x.l}; }
__device__ __forceinline__ double df_double(df x) { return (double)x.h + (double)x.l; }

// The leading 48 bits of a double as a double-float, on the integer units (an FP64 conversion costs
// as much as an FP64 operation): the upper 24 bits of the significand are the high part (truncated),
// the other 29, rounded to 24, the low part.  Exact exponents for 2^-73 <= |v| < 2^128; smaller
// values lose the low part, infinities and NaN stay what they are.  k: the pair of 2^-k v (|k| <= 608).
__device__ __forceinline__ df df_split(double v, int k = 0) {
  const long long u = __double_as_longlong(v);
  const unsigned hi = (unsigned)((unsigned long long)u >> 32), lo = (unsigned)u;
  const int e = (int)((hi >> 20) & 0x7ffu);
  const unsigned sign = hi & 0x80000000u;
  const int eh = min(max(e - 896 - k, 0), 255);
  const unsigned m = (hi << 3 & 0x7fffffu) | (lo >> 29);
  const float h = __uint_as_float(sign | ((unsigned)eh << 23) | m);
  const int el = eh == 255 ? 0 : max(e - 948 - k, 0);
  const float l = __fmul_rn((float)(lo & 0x1fffffffu), __uint_as_float(sign | ((unsigned)el << 23)));
  return {h, l};
}

// Butterfly reduce-scatter of M double-floats over a warp, as Butterfly in mq_device.cuh: on return
// v[0] holds the warp total of value index `base` when c >= 1.
template <int M, int O>
struct DfButterfly {
  static __device__ __forceinline__ void run(df* v, int lane, int& base, int& c) {
    constexpr int H = (M + 1) / 2;
    const bool b = (lane & O) != 0;
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const df lo = v[i], hi = (H + i < M) ? v[H + i] : df{0.0f, 0.0f};
      const df send = b ? lo : hi, keep = b ? hi : lo;
      v[i] = df_add(keep, df{__shfl_xor_sync(0xffffffffu, send.h, O), __shfl_xor_sync(0xffffffffu, send.l, O)});
    }
    if (b) {
      base += H;
      c = max(0, c - H);
    } else {
      c = min(c, H);
    }
    DfButterfly<H, O / 2>::run(v, lane, base, c);
  }
};
template <int M>
struct DfButterfly<M, 0> {
  static __device__ __forceinline__ void run(df*, int, int&, int&) {}
};

}  // namespace dev
}  // namespace mq

// Centroid coefficients a = a0 + Y Psi on the 5th-generation tensor cores (tcgen05, sm_103a),
// accurate to FP64 rounding of the terms.
//
// The dense contraction of eq. coeff (samples x truncation) x (truncation x triangles) is split
// into exact BF16 integer slices (an Ozaki-type splitting):
//   y   in [-1/2, 1/2):  y   = sum_{p<7} Y_p 2^{-8(p+1)}  + r,  |r| <= 2^-57,  Y_p integers in [-128, 128]
//   psi in [-1, 1]:      psi = sum_{q<7} P_q 2^{-7-8q}    + r,  |r| <= 2^-64,  P_q integers in [-128, 128]
// (a table is scaled by 2^e first, e chosen from its largest term factor so that |2^e psi| <= 1
// with the most bits kept; the result is scaled back by the exact factor 2^-e)
// Integers of magnitude <= 256 are exact in BF16, products of two are exact in the FP32
// accumulator, and every accumulated sum stays an integer below 2^24 (K is processed in chunks of
// at most 128 and the products are grouped by g = p + q, at most 7 per group: 7 * 128 * 2^14 <
// 2^24), so each group sum
//   S_g = sum_{p+q=g} sum_{j in chunk} Y_p[b][j] P_q[t][j]
// is EXACT whatever the accumulation order of the tensor core.  Groups g <= 6 are kept (28 slice
// products): a = a0 + sum_chunks sum_g 2^{-15-8g} S_g, the group sums combined in 64-bit
// integers and rounded once to FP64.  Dropped products (g >= 7) and slice remainders are below 2^-56 per term: the result
// matches an FP64 GEMM to a few units of FP64 rounding.
//
// Kernel (persistent, one CTA of 18 warps per SM): each CTA walks 128-sample x 64-triangle output
// tiles.  Per 16-wide K step one thread of warp 17 has the tensor memory accelerator load the seven
// A slices (128 x 16) and the seven B slices (64 x 16) into one of five shared-memory stages (slices
// are stored K-blocked, [slice][K/8][row][8], so one 4-D box lands directly in the canonical
// no-swizzle K-major layout of 8 x 16-byte core matrices).  One thread of warp 16 waits for a stage
// and issues ten tcgen05.mma (kind::f16, BF16 x BF16 -> FP32, M = 128, N = 64 .. 256, K = 16: each A
// slice against up to four B slices at once) into seven TMEM accumulators (64 columns each), and
// commits them to the stage's "empty" mbarrier.  After
// every 128-wide K chunk the sixteen other warps read the accumulators with tcgen05.ld (warp w: TMEM
// lanes 32 (w mod 4).., columns 16 (w div 4)..), hand the accumulators back to warp 16 as soon as
// their last load has arrived, and finish the tile -- rounding and stores -- while the tensor cores
// work on the next one.
//
// The fold is the kernel's cost: at K = 48 the products of a tile take ~3,300 clocks.  The whole sum
// a0 + sum_g 2^{-15-8g} S_g is formed in 64-bit fixed point (resolution 2^{s-63-e}, 2^{s-e} four times
// the largest |a| the terms allow for |y| <= 1/2) and rounded to FP64 once, about 32 instructions per output;
// rounding the chunk exactly from 128 bits and adding a0 in FP64 took ~300 and eight warps.
// Measured with the form for short contractions below, 64 samples on mesh 1/1024 with 1,024 terms (134 M
// outputs, 0.16 ms to write them): 1.8 ms before, 0.5 ms now.
// Contractions whose a0 is beyond about 2^8 times the largest term, or below 2^-10 of it, keep the 128-bit form.  Every wait is
// bounded; a timeout sets an error word, stops the issuing of new work, drains what is in flight
// and frees the tensor memory.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "mq_internal.h"

namespace mq {
namespace {

constexpr int kSlices = 7;   // slices per operand
constexpr int kGroups = 7;   // kept groups g = p + q
constexpr int kTM = 128;     // samples per tile (TMEM lanes)
constexpr int kTN = 64;      // triangles per tile
constexpr int kTK = 16;      // K per MMA (one pipeline step)
constexpr int kChunk = 128;  // K per exact accumulation chunk
constexpr int kStepsPerChunk = kChunk / kTK;
constexpr int kWide = 256 / kTN;  // B slices per MMA (N <= 256)
constexpr int kStages = 5;   // shared-memory pipeline depth (5 x 42 KB)
constexpr int kEpiWarps = 16;                      // fold and store
constexpr int kTcThreads = 32 * (kEpiWarps + 2);  // + the MMA warp and the TMA warp
constexpr int kTmemCols = 512;  // 7 groups x 64 columns = 448 used
constexpr uint32_t kABytes = kSlices * kTM * kTK * 2;  // 28 KB per stage
constexpr uint32_t kBBytes = kSlices * kTN * kTK * 2;  // 14 KB per stage
constexpr long kSpinLimit = 1L << 22;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: no swizzle, K-major core matrices of 8 rows x 16 bytes;
// lbo = byte distance between core matrices adjacent in K, sbo = between 8-row groups
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version of the 5th-generation tensor core
  return d;                // base offset 0, layout type 0 (no swizzle)
}

// instruction descriptor, kind::f16: D = F32, A = B = BF16, both K-major, M = 128, N columns
__host__ __device__ constexpr uint32_t instr_desc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTM >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint64_t* mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(mbar))
               : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t* mbar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(count) : "memory");
}

// arrive once and expect `bytes` of asynchronous (TMA) transfers on the barrier's current phase
__device__ __forceinline__ void mbar_arrive_expect(uint64_t* mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mbar)), "r"(bytes) : "memory");
}

// bounded wait for the phase with the given parity; false when the limit ran out
__device__ __forceinline__ bool mbar_wait(uint64_t* mbar, uint32_t parity) {
  const uint32_t addr = smem_u32(mbar);
  for (long i = 0; i < kSpinLimit; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// 4-D tiled TMA load of one box into shared memory, completing on an mbarrier
__device__ __forceinline__ void tma_load4(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                          uint64_t* mbar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
      "[%6];" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(mbar))
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 8 consecutive TMEM columns of this thread's lane, without waiting: the registers are valid
// only after tmem_wait on them (several loads can then share one wait)
__device__ __forceinline__ void tmem_ld8_async(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

// waits for this thread's outstanding TMEM loads; the registers are passed through so that no use
// of them can be scheduled before the wait
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
               :
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(mbar)) : "memory");
}

// four doubles to a 32-byte aligned address in one store (a whole memory sector)
__device__ __forceinline__ void st_sector(double* p, const double (&v)[4]) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3])
               : "memory");
}

// ---------------------------------------------------------------------------------------------
// slicing.  out layout [slice][kpad / 8][rows_pad][8] (blocks of eight K values per row, the row
// blocks back to back): a TMA box of 8 x rows x 2 x 7 is then one K step of all slices, in the
// core-matrix layout the MMA reads.  Zero padding beyond rows / k.
__global__ void k_slice_rows(const double* __restrict__ src, int rows, int k, size_t row_stride, size_t col_stride,
                             double scale, int rows_pad, int kpad, __nv_bfloat16* __restrict__ out) {
  const size_t tot = (size_t)rows_pad * kpad;
  for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < tot; q += (size_t)gridDim.x * blockDim.x) {
    const int e = (int)(q & 7);
    const size_t rb = q >> 3;  // jb * rows_pad + r
    const int r = (int)(rb % rows_pad), j = (int)(rb / rows_pad) * 8 + e;
    double v = (r < rows && j < k) ? src[(size_t)r * row_stride + (size_t)j * col_stride] * scale : 0.0;
#pragma unroll
    for (int p = 0; p < kSlices; ++p) {
      const double s = rint(v);
      out[(size_t)p * tot + q] = __float2bfloat16_rn((float)s);
      v = (v - s) * 256.0;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Separable evaluation (families whose terms are c_t sin(pi k1_t x1) sin(pi k2_t x2) with few
// distinct k1, like the workload family, where k1 <= ~2 sqrt(s)).  On one plane of triangles
// (lower or upper: the centroid abscissa x_i depends only on the cell column i, the ordinate y_j
// only on the cell row j)
//     a[b][j][i] = a0 + sum_{k1} T[b][j][k1] sin(pi k1 x_i),
//     T[b][j][k1] = sum_{t < K, k1_t = k1} Y[b][t] c_t sin(pi k2_t y_j),
// the same sum as eq. coeff_s grouped by k1.  Stage 1 forms T in fixed point on the integer units (B n K
// products for both planes together) and writes its exact BF16 slices; stage 2 is the tensor-core
// kernel below with rows (b, j), columns i and K = the padded count of k1 values: 2 B n^2 K1
// products per plane instead of 2 B n^2 K.

// centroid numerators over 3n: abscissa of column i, ordinate of row j, per plane
__device__ __forceinline__ int cx_num(int i, int plane) { return 3 * i + (plane == 0 ? 2 : 1); }
__device__ __forceinline__ int cy_num(int j, int plane) { return 3 * j + (plane == 0 ? 1 : 2); }

// A fixed-point value v 2^-60 of stage 1 as two parts, v = x 2^30 + y with |y| <= 2^29
__device__ __forceinline__ int2 fixed_parts(long long v) {
  const int lo = (int)(((v + (1LL << 29)) & ((1LL << 30) - 1)) - (1LL << 29));
  return make_int2((int)((v - lo) >> 30), lo);
}

// sy[k][j] = sin(pi k y_j) on the lower plane, k = 0..kmax, j < n (on the upper plane y_{n-1-j} is 1 - y_j
// of the lower one, so its sines are these times (-1)^{k+1})
__global__ void k_sep_sy(int n, int kmax, int2* __restrict__ sy) {
  const size_t tot = (size_t)(kmax + 1) * n;
  for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < tot; q += (size_t)gridDim.x * blockDim.x) {
    const int k = (int)(q / n), j = (int)(q % n);
    sy[q] = fixed_parts(__double2ll_rn(sinpi((double)((long)k * cy_num(j, 0) % (6L * n)) / (double)(3 * n)) * 1152921504606846976.0));
  }
}

// sx[i][e] = sin(pi (e+1) x_i) for e + 1 <= k1max, 0 beyond (kpad columns)
__global__ void k_sep_sx(int n, int plane, int k1max, int kpad, double* __restrict__ sx) {
  const size_t tot = (size_t)n * kpad;
  for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < tot; q += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(q / kpad), e = (int)(q % kpad);
    sx[q] = e + 1 <= k1max ? sinpi((double)((long)(e + 1) * cx_num(i, plane) % (6L * n)) / (double)(3 * n)) : 0.0;
  }
}

// The factors of stage 1, formed once per sample in list order: yc[b][i] = s60 Y[b][t] c_t of the term t =
// list[i].x (s60 = scale 2^60; zero for t >= K), and the end kend[v] of the terms below K in sublist v
// (each sublist is in increasing t)
__global__ void k_sep_yc(const double* __restrict__ Y, int ldy, int B, int K, const double* __restrict__ cj,
                         const int2* __restrict__ list, const int* __restrict__ start, int nlist, int nsub, double s60,
                         int2* __restrict__ yc, int* __restrict__ kend) {
  const size_t tot = (size_t)B * nlist;
  const size_t g = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (size_t q = g; q < tot; q += (size_t)gridDim.x * blockDim.x) {
    const int b = (int)(q / nlist), t = list[q % nlist].x;
    yc[q] = t < K ? fixed_parts(__double2ll_rn(Y[(size_t)b * ldy + t] * cj[t] * s60)) : make_int2(0, 0);
  }
  if (g < (size_t)nsub) {
    int lo = start[g], hi = start[g + 1];
    while (lo < hi) {
      const int mid = (lo + hi) / 2;
      if (list[mid].x < K)
        lo = mid + 1;
      else
        hi = mid;
    }
    kend[g] = lo;
  }
}

// 8 BF16 digits per slice from 8 values W = sum_p d_p 2^{8(6-p)}: with 0x80 added to each of the six low
// bytes, those bytes minus 128 are the digits d_1 .. d_6 and the rest is d_0.  A byte becomes a float
// by its place in the significand of 2^23 (no conversion instruction); digits are exact in BF16.
__device__ __forceinline__ void put_digits(const long long (&W)[8], size_t sstride, size_t at,
                                           __nv_bfloat16* __restrict__ out) {
  unsigned lo[8], hi[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const unsigned long long u = (unsigned long long)W[e] + 0x808080808080ull;
    lo[e] = (unsigned)u, hi[e] = (unsigned)(u >> 32);
  }
#pragma unroll
  for (int p = 0; p < kSlices; ++p) {
    float f[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (p == 0) {
        f[e] = __int_as_float(0x4B400000 + ((int)hi[e] >> 16)) - 12582912.0f;
      } else {
        const int byte = 6 - p;  // byte of u holding d_p
        f[e] = __uint_as_float(__byte_perm(byte < 4 ? lo[e] : hi[e], 0x4B000000u, 0x7650u | (byte & 3))) - 8388736.0f;
      }
    }
    uint4 v;
    v.x = __byte_perm(__float_as_uint(f[0]), __float_as_uint(f[1]), 0x7632);
    v.y = __byte_perm(__float_as_uint(f[2]), __float_as_uint(f[3]), 0x7632);
    v.z = __byte_perm(__float_as_uint(f[4]), __float_as_uint(f[5]), 0x7632);
    v.w = __byte_perm(__float_as_uint(f[6]), __float_as_uint(f[7]), 0x7632);
    *reinterpret_cast<uint4*>(out + (size_t)p * sstride + at) = v;
  }
}

// Stage 1: T[m = b n + j][k1 - 1] of both planes, written as the 7 BF16 slices of 256 scale T in the
// layout of k_slice_rows ([7][kpad/8][rows_pad][8]); one thread per (row, group of 8 k1 values).
// Sublist 2 (k1 - 1) + c of list holds the terms (t, k2) of k1 with even (c = 0) or odd (c = 1) k2: their
// sums give both planes at once, T = odd + even on the lower plane at row j, odd - even on the
// upper plane at row n - 1 - j.  Factors carry 2^-60 (sum |scale y c| <= 1/2 for |y| <= 1/2); a product is
// three 32 x 32 -> 64-bit multiply-adds (the low parts' own product is below 2^-62).
// The FP64 form of this kernel (one FP64 multiply-add per product and plane, at GB300's FP64 issue
// rate) took 380 us for 64 samples on mesh 1/1024 with 1,024 terms, this one 106 us.
__global__ void __launch_bounds__(256) k_sep_stage1(const int2* __restrict__ yc, int B, int n, int nlist, int kpad,
                                                    const int* __restrict__ start, const int* __restrict__ kend,
                                                    const int2* __restrict__ list, const int2* __restrict__ sy,
                                                    int rows_pad, __nv_bfloat16* __restrict__ out0,
                                                    __nv_bfloat16* __restrict__ out1) {
  const size_t tot = (size_t)rows_pad * (kpad / 8);
  const size_t sstride = (size_t)rows_pad * kpad;
  const int rows = B * n;
  for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < tot; q += (size_t)gridDim.x * blockDim.x) {
    const int m = (int)(q % rows_pad), kg = (int)(q / rows_pad);
    const int b = m / n, j = m % n;
    const int2* __restrict__ yb = yc + (size_t)b * nlist;
    const int2* __restrict__ sj = sy + j;
    long long W0[8], W1[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      long long T[2] = {0, 0};
#pragma unroll
      for (int par = 0; par < 2; ++par) {
        const int v = 2 * (kg * 8 + e) + par;
        const int i1 = m < rows ? kend[v] : 0;
        long long h = 0, c = 0;  // high products, cross products 2^-30
        for (int i = start[v]; i < i1; i += 4) {
          int2 y[4], sv[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int ii = min(i + k, i1 - 1);
            y[k] = yb[ii];
            sv[k] = sj[(size_t)list[ii].y * n];
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (i + k >= i1) y[k] = make_int2(0, 0);
            h += (long long)y[k].x * sv[k].x;
            c += (long long)y[k].x * sv[k].y;
            c += (long long)y[k].y * sv[k].x;  // eight cross products below 2^60 at most
          }
          h += c >> 30;
          c &= (1LL << 30) - 1;
        }
        T[par] = h;
      }
      W0[e] = (T[1] + T[0] + 8) >> 4;  // units of 2^-56
      W1[e] = (T[1] - T[0] + 8) >> 4;
    }
    put_digits(W0, sstride, ((size_t)kg * rows_pad + m) * 8, out0);
    put_digits(W1, sstride, ((size_t)kg * rows_pad + (m < rows ? m - j + (n - 1 - j) : m)) * 8, out1);
  }
}

// (hi 2^24 + lo) 2^e rounded once to the nearest double (ties to even), in integer arithmetic:
// the exact sum of a chunk's group sums, |hi| < 2^56, |lo| < 2^40.  GB300 issues FP64 at 1/64 of
// the FP32 rate; the conversions and the fused multiply-add of the FP64 fold cost more issue time
// than this on the integer units.  The result is finite and normal for every e the tables use.
__device__ __forceinline__ double exact_fold(long long hi, long long lo, int e) {
  const __int128 v = ((__int128)hi << 24) + (__int128)lo;
  if (v == 0) return 0.0;
  const bool neg = v < 0;
  unsigned __int128 m = neg ? (unsigned __int128)(-v) : (unsigned __int128)v;
  const unsigned long long mh = (unsigned long long)(m >> 64), ml = (unsigned long long)m;
  const int lz = mh ? __clzll((long long)mh) : 64 + __clzll((long long)ml);
  m <<= lz;  // leading one at bit 127
  const unsigned long long top = (unsigned long long)(m >> 64), rest = (unsigned long long)m;
  unsigned long long mant = top >> 11;  // 53 bits
  const unsigned long long rb = top & 0x7FFull;  // the next 11 bits; rest holds the ones below
  mant += (rb > 0x400ull) || (rb == 0x400ull && (rest != 0ull || (mant & 1ull)));
  int ex = 127 - lz + e;
  if (mant >> 53) {
    mant >>= 1;
    ++ex;
  }
  const unsigned long long bits = ((unsigned long long)neg << 63) | ((unsigned long long)(ex + 1023) << 52) |
                                  (mant & ((1ull << 52) - 1));
  return __longlong_as_double((long long)bits);
}

// v 2^e rounded once to the nearest double (ties to even); the result is normal for every e in use.
// positive: v has a bit in its upper word and is not negative, as every valid coefficient is.
__device__ __forceinline__ double fixed_positive(unsigned long long v, int e) {
  unsigned hi = (unsigned)(v >> 32), lo = (unsigned)v;
  const int lz = __clz((int)hi);
  hi = __funnelshift_l(lo, hi, lz);  // leading one at bit 31
  lo <<= lz;
  const unsigned ml = __funnelshift_r(lo, hi, 11);
  const unsigned round = ((lo & 0x7FFu) + 0x3FFu + (ml & 1u)) >> 11;
  // the leading one of the significand (or the carry of the rounding) adds to the exponent field
  const unsigned long long bits =
      (((unsigned long long)(((unsigned)(e + 63 + 1022 - lz) << 20) + (hi >> 11)) << 32) | ml) + round;
  return __longlong_as_double((long long)bits);
}
__device__ __forceinline__ double fixed_to_double(long long v, int e) {
  if (v == 0) return 0.0;
  unsigned long long u = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const bool small = (u >> 32) == 0;
  const double d = fixed_positive(small ? u << 32 : u, small ? e - 32 : e);
  return v < 0 ? -d : d;
}
// N outputs at once: the common case without branches, so that the outputs' chains overlap
template <int N>
__device__ __forceinline__ void fixed_to_doubles(const long long (&v)[N], int e, double (&d)[N]) {
  bool ok = true;
#pragma unroll
  for (int i = 0; i < N; ++i) ok = ok && (int)((unsigned long long)v[i] >> 32) > 0;
  if (ok) {
#pragma unroll
    for (int i = 0; i < N; ++i) d[i] = fixed_positive((unsigned long long)v[i], e);
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) d[i] = fixed_to_double(v[i], e);
  }
}
// v 2^-e rounded to an integer (|v 2^-e| < 2^63): the fixed-point image of a zeroth term
__device__ __forceinline__ long long double_to_fixed(double v, int e) {
  const long long b = __double_as_longlong(v);
  const int ex = (int)((b >> 52) & 0x7FF);
  if (ex == 0) return 0;  // zero (a subnormal is far below the resolution)
  const unsigned long long m = ((unsigned long long)b & ((1ull << 52) - 1)) | (1ull << 52);
  const int sh = ex - 1075 - e;  // v = m 2^{ex - 1075}
  unsigned long long r;
  if (sh >= 0)
    r = m << min(sh, 63);
  else
    r = sh < -54 ? 0ull : (m + (1ull << (-sh - 1))) >> -sh;
  return b < 0 ? -(long long)r : (long long)r;
}

struct alignas(1024) TcSmem {
  __nv_bfloat16 a[kStages][kSlices * kTM * kTK];  // [slice][K half][128 rows][8]
  __nv_bfloat16 b[kStages][kSlices * kTN * kTK];  // [K half][slice][64 rows][8]: the slices' rows contiguous
  uint64_t full[kStages];   // TMA bytes of a stage landed
  uint64_t empty[kStages];  // the MMAs that read a stage completed
  uint64_t accf;            // the MMAs of a K chunk completed (accumulators readable)
  uint64_t acce;            // the fold warps hold the chunk in registers (accumulators free)
  uint32_t tmem_base;
  uint32_t loads, uses, commits;  // K steps loaded, consumed, committed (for the drain after an error)
  volatile int err;
};

// Output placement: element (row b, column t) goes to out[row_off(b) + t] with row_off(b) = b nT,
// or, with mdiv > 0, (b / mdiv) m_hi + (b mod mdiv) m_lo (rows that index (sample, mesh row)
// pairs of a coefficient field).  Rows come in tiles of 128, columns in tiles of 64.
struct TcOut {
  double* out;
  int mdiv;
  long long m_hi, m_lo;
  int cols_fast;  // tile order: 0 row tiles fastest (tiles sharing a column tile run together), 1 columns
};

// Domain: |y| <= 1 (the lattice points lie in [-1/2, 1/2)): the leading digit of y is then at most 256, the
// largest one exact in BF16, all others at most 128, and a group sum over 16 T terms is bounded by
//   |S_g| <= (g + 2) 16 T 2^14   (at most 2^24, exact in FP32, for the 128 terms of a chunk).
// One output's group sums in units of 2^fs, added to w modulo 2^64:
//   sum_g S_g 2^{8(6-g)-fs} = A 2^{40-fs} + B 2^{24-fs} + S_4 2^{16-fs} + D,
//   A = S_0 256 + S_1, B = S_2 256 + S_3, D = S_5 2^{8-fs} + floor(S_6 2^-fs) (1 <= fs <= 8);
// A and D stay below 2^31, B up to 80 terms (a whole chunk: 64 bits).
__device__ __forceinline__ int group_sum(uint32_t r) { return __float2int_rn(__uint_as_float(r)); }
// the same for |S_g| <= 2^22 without a conversion instruction (those run at an eighth of the rate): the
// integer from the significand of 1.5 2^23 + S_g
constexpr int small_groups(int T) {  // the groups (of the first five) that this holds for
  int g = 0;
  while (g < 5 && ((g + 2) * 16 * T) << 14 <= 1 << 22) ++g;
  return g;
}
template <bool SMALL>
__device__ __forceinline__ int group_sum_if(uint32_t r) {
  return SMALL ? __float_as_int(__uint_as_float(r) + 12582912.0f) - 0x4B400000 : group_sum(r);
}
template <typename I>
__device__ __forceinline__ long long fold_fixed(int A, I Bv, int s4, int s5, int s6, int fs, long long w) {
  long long x = (long long)s4 * (1 << (16 - fs)) + w;
  x = (long long)(s5 * (1 << (8 - fs)) + (s6 >> fs)) * 1 + x;
  x = (long long)Bv * (1 << (24 - fs)) + x;
  const unsigned xh = (unsigned)((unsigned long long)x >> 32) + (unsigned)A * (1u << (8 - fs));
  return (long long)(((unsigned long long)xh << 32) | (unsigned)x);
}

// start of output row b (the row of tile column t0)
__device__ __forceinline__ double* out_row(const TcOut& O, int nT, int b, int t0) {
  return O.out + t0 + (O.mdiv > 0 ? (size_t)(b / O.mdiv) * (size_t)O.m_hi + (size_t)(b % O.mdiv) * (size_t)O.m_lo
                                  : (size_t)b * nT);
}

// The short contraction (K <= 80: the separable stage, short truncations), fixed point: the same
// products and fold with the A operand resident.  A CTA takes a contiguous range of tiles of 128
// samples x 32 triangles, columns fastest, and keeps all K steps of its sample rows in shared memory
// (28 KB each) while the triangles' slices stream by, one stage per tile; the 7 x 32 accumulator
// columns fit the tensor memory twice, so the sixteen fold warps work on one tile while warp 16 issues
// the products of the next.  Streaming both operands with one set of 7 x 64 columns moved
// 172 KB per tile through L2 at K = 64 (7.5 TB/s, its limit) and left the tensor cores idle during the fold.
constexpr int kRN = 32;          // triangles per tile
constexpr int kResSteps = 5;     // K steps at most
constexpr int kResStages = 6;    // triangle stages at most
constexpr int kResSmem = 220 * 1024;
constexpr uint32_t kRBytes = kSlices * kRN * kTK * 2;  // 7 KB per K step

struct ResSmem {
  uint64_t full[kResStages], empty[kResStages];  // a tile's triangle slices landed / were consumed
  uint64_t afull;                                // the sample slices of a row tile landed
  uint64_t accf[2], acce[2];                     // accumulator set computed / in the fold warps' registers
  uint32_t tmem_base;
  uint32_t loads, uses, commits, aloads, auses;  // for the drain after an error
  volatile int err;
};

// SMALL: groups g < SMALL hold sums of at most 2^22 (small_groups of the largest T)
template <int SMALL>
__global__ void __launch_bounds__(kTcThreads, 1)
    k_coef_res(const __grid_constant__ CUtensorMap tmY, const __grid_constant__ CUtensorMap tmP, int B, int nT, int T,
               int nst, int ntn, int ntiles, double a0, TcOut O, int* __restrict__ err_flag,
               const double* __restrict__ base, int pexp, int fs) {
  extern __shared__ __align__(1024) char dyn[];
  char* sm = (char*)(((uintptr_t)dyn + 1023) & ~(uintptr_t)1023);  // A: T x 28 KB, then nst stages of T x 7 KB
  __shared__ ResSmem S;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int first = (int)((long)ntiles * blockIdx.x / gridDim.x), last = (int)((long)ntiles * (blockIdx.x + 1) / gridDim.x);
  char* sb = sm + (size_t)T * kABytes;
  const uint32_t stage_bytes = (uint32_t)T * kRBytes;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem_base)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < kResStages; ++i) {
      mbar_init(&S.full[i], 1);
      mbar_init(&S.empty[i], 1);
    }
    mbar_init(&S.afull, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&S.accf[i], 1);
      mbar_init(&S.acce[i], kEpiWarps);
    }
    S.loads = S.uses = S.commits = S.aloads = S.auses = 0;
    S.err = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem_base;
  if (warp == kEpiWarps + 1) {
    // ---- loads
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmY) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmP) : "memory");
      int row = -1;
      uint32_t u = 0;
      for (int tile = first; tile < last && !S.err; ++tile, ++u) {
        const uint32_t st = u % (uint32_t)nst;
        const int tm = tile / ntn, tn = tile % ntn;
        if (tm != row) {
          // the products of the previous row tile must be done: those of its last tile are
          if (row >= 0 && !mbar_wait(&S.empty[(u - 1) % (uint32_t)nst], ((u - 1) / (uint32_t)nst) & 1)) {
            S.err = 1;
            break;
          }
          row = tm;
          mbar_arrive_expect(&S.afull, (uint32_t)T * kABytes);
          for (int ks = 0; ks < T; ++ks) tma_load4(sm + (size_t)ks * kABytes, &tmY, 0, tm * kTM, 2 * ks, 0, &S.afull);
          ++S.aloads;
        }
        // the stage's previous tile must have been consumed
        if (u >= (uint32_t)nst && !mbar_wait(&S.empty[st], (u / (uint32_t)nst - 1) & 1)) {
          S.err = 1;
          break;
        }
        mbar_arrive_expect(&S.full[st], stage_bytes);
        for (int ks = 0; ks < T; ++ks)
          tma_load4(sb + (size_t)st * stage_bytes + (size_t)ks * kRBytes, &tmP, 0, tn * kRN, 0, 2 * ks, &S.full[st]);
        S.loads = u + 1;
      }
    }
  } else if (warp == kEpiWarps) {
    // ---- products
    if (lane == 0) {
      int row = -1;
      uint32_t u = 0, rows = 0;
      for (int tile = first; tile < last && !S.err; ++tile, ++u) {
        const uint32_t st = u % (uint32_t)nst, set = u & 1;
        const int tm = tile / ntn;
        if (tm != row) {
          row = tm;
          if (!mbar_wait(&S.afull, rows & 1)) {
            S.err = 1;
            break;
          }
          S.auses = ++rows;
        }
        // the set's previous tile must be in the fold warps' registers
        if ((u >= 2 && !mbar_wait(&S.acce[set], (u / 2 - 1) & 1)) || !mbar_wait(&S.full[st], (u / (uint32_t)nst) & 1)) {
          S.err = 1;
          break;
        }
        S.uses = u + 1;
        tc_fence_after();
        const uint32_t abase = smem_u32(sm), bbase = smem_u32(sb) + st * stage_bytes, acc = tmem + set * 256;
        for (int ks = 0; ks < T; ++ks) {
          // A slice p times the B slices 0 .. 6 - p: the groups p .. 6, side by side
#pragma unroll
          for (int p = 0; p < kSlices; ++p) {
            const uint64_t ad = smem_desc(abase + ks * kABytes + p * (kTM * kTK * 2), kTM * 16, 128);
            const uint64_t bd = smem_desc(bbase + ks * kRBytes, kSlices * kRN * 16, 128);
            mma_bf16(acc + (uint32_t)(p * kRN), ad, bd, instr_desc((kGroups - p) * kRN), (ks > 0 || p > 0) ? 1u : 0u);
          }
        }
        mma_commit(&S.empty[st]);
        mma_commit(&S.accf[set]);
        S.commits = u + 1;
      }
    }
  } else {
    // ---- fold and store: warp w takes lanes 32 (w mod 4).. and columns 8 (w div 4)..
    const int q4 = warp & 3, cg = warp >> 2;
    const int fe = fs - 63 - pexp;
    const long long f0 = base ? 0 : double_to_fixed(a0, fe);
    uint32_t u = 0;
    int tm = first / ntn, tn = first % ntn;
    double* o = nullptr;  // this lane's output row at column 8 (w div 4) of the column tile tn
    for (int tile = first; tile < last; ++tile, ++u) {
      const uint32_t set = u & 1;
      // (the whole warp leaves or stays: the tensor-memory loads below need it converged)
      if (__any_sync(0xffffffffu, S.err || !mbar_wait(&S.accf[set], (u / 2) & 1))) {
        S.err = 1;
        break;
      }
      tc_fence_after();
      const uint32_t tcol = tmem + ((uint32_t)(q4 * 32) << 16) + set * 256 + (uint32_t)(cg * 8);
      uint32_t r[kGroups][8];
#pragma unroll
      for (int g = 0; g < kGroups; ++g) tmem_ld8_async(tcol + (uint32_t)(g * kRN), r[g]);
#pragma unroll
      for (int g = 0; g < kGroups; ++g) tmem_wait(r[g]);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&S.acce[set]);  // the accumulators may be overwritten
      const int t0 = tn * kRN + cg * 8;
      if (u == 0 || tn == 0) {
        const int b = tm * kTM + q4 * 32 + lane;
        o = b < B ? out_row(O, nT, b, t0) : nullptr;
      }
      long long w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        w[i] = fold_fixed(group_sum_if<(SMALL > 0)>(r[0][i]) * 256 + group_sum_if<(SMALL > 1)>(r[1][i]),
                          group_sum_if<(SMALL > 2)>(r[2][i]) * 256 + group_sum_if<(SMALL > 3)>(r[3][i]),
                          group_sum_if<(SMALL > 4)>(r[4][i]), group_sum(r[5][i]), group_sum(r[6][i]), fs, f0);
      if (base) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (t0 + i < nT) w[i] = (long long)((unsigned long long)w[i] + (unsigned long long)double_to_fixed(base[t0 + i], fe));
      }
      double d[8];
      fixed_to_doubles<8>(w, fe, d);
      if (o) {
        if (t0 + 8 <= nT && ((uintptr_t)o & 31) == 0) {
          st_sector(o, *reinterpret_cast<const double(*)[4]>(d));
          st_sector(o + 4, *reinterpret_cast<const double(*)[4]>(d + 4));
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (t0 + i < nT) o[i] = d[i];
        }
        o += kRN;
      }
      if (++tn == ntn) {
        tn = 0;
        ++tm;
      }
      __syncwarp();
    }
  }
  __syncthreads();
  if (tid == 0) {
    if (S.err) {
      atomicOr(err_flag, 1);
      // drain the loads that no product consumed
      for (uint32_t u = S.uses; u < S.loads; ++u) mbar_wait(&S.full[u % (uint32_t)nst], (u / (uint32_t)nst) & 1);
      for (uint32_t u = S.auses; u < S.aloads; ++u) mbar_wait(&S.afull, u & 1);
    }
    // and the last products of every stage
    for (uint32_t u = S.commits > (uint32_t)nst ? S.commits - (uint32_t)nst : 0; u < S.commits; ++u)
      mbar_wait(&S.empty[u % (uint32_t)nst], (u / (uint32_t)nst) & 1);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

// a[b][t] = a0 + sum_j y[b][j] psi[j][t], b < B, t < nT (with base: base[t] in place of a0).
// Tiles: tm = tile mod ntm (128 samples), tn = tile div ntm (64 triangles), or the transposed
// order; CTA c takes tiles c, c + grid, ...  Kpad: K of the Y slices.  FIXED: the sum in 64-bit fixed
// point of resolution 2^{fs - 63 - pexp} (1 <= fs <= 8); otherwise chunk by chunk in FP64.
template <bool FIXED>
__global__ void __launch_bounds__(kTcThreads, 1)
    k_coef_tc(const __grid_constant__ CUtensorMap tmY, const __grid_constant__ CUtensorMap tmP, int B, int nT, int Kpad,
              int ntm, int ntiles, double a0, TcOut O, int* __restrict__ err_flag, const double* __restrict__ base,
              int pexp, int fs) {
  const int ntn = ntiles / ntm;
  auto coords = [&](int tile, int& tm, int& tn) {
    if (O.cols_fast) {
      tm = tile / ntn;
      tn = tile % ntn;
    } else {
      tm = tile % ntm;
      tn = tile / ntm;
    }
  };
  extern __shared__ __align__(1024) char dyn[];
  TcSmem& S = *reinterpret_cast<TcSmem*>(((uintptr_t)dyn + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int T = Kpad / kTK;  // K steps per tile
  const int nchunk = (T + kStepsPerChunk - 1) / kStepsPerChunk;
  const int my_tiles = (int)blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  const uint32_t U = (uint32_t)my_tiles * (uint32_t)T;  // K steps of this CTA
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem_base)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&S.full[i], 1);
      mbar_init(&S.empty[i], 1);
    }
    mbar_init(&S.accf, 1);
    mbar_init(&S.acce, kEpiWarps);
    S.loads = S.uses = S.commits = 0;
    S.err = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem_base;
  if (warp == kEpiWarps + 1) {
    // ---- loads
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmY) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmP) : "memory");
      uint32_t u = 0;
      for (int ti = 0; ti < my_tiles && !S.err; ++ti) {
        int tm, tn;
        coords((int)blockIdx.x + ti * (int)gridDim.x, tm, tn);
        for (int ks = 0; ks < T && !S.err; ++ks, ++u) {
          const uint32_t st = u % kStages;
          // the stage's previous step must have been consumed
          if (u >= (uint32_t)kStages && !mbar_wait(&S.empty[st], (u / kStages - 1) & 1)) {
            S.err = 1;
            break;
          }
          mbar_arrive_expect(&S.full[st], kABytes + kBBytes);
          tma_load4(S.a[st], &tmY, 0, tm * kTM, 2 * ks, 0, &S.full[st]);
          tma_load4(S.b[st], &tmP, 0, tn * kTN, 0, 2 * ks, &S.full[st]);
          S.loads = u + 1;
        }
      }
    }
  } else if (warp == kEpiWarps) {
    // ---- products
    if (lane == 0) {
      uint32_t u = 0, chunk = 0;
      for (int ti = 0; ti < my_tiles && !S.err; ++ti) {
        for (int kc = 0; kc < T && !S.err; kc += kStepsPerChunk, ++chunk) {
          const int kend = min(T, kc + kStepsPerChunk);
          // the accumulators of the previous chunk must be in the fold warps' registers
          if (chunk >= 1 && !mbar_wait(&S.acce, (chunk - 1) & 1)) {
            S.err = 1;
            break;
          }
          tc_fence_after();
          for (int ks = kc; ks < kend; ++ks, ++u) {
            const uint32_t st = u % kStages;
            if (S.err || !mbar_wait(&S.full[st], (u / kStages) & 1)) {
              S.err = 1;
              break;
            }
            S.uses = u + 1;
            tc_fence_after();
            const uint32_t abase = smem_u32(S.a[st]), bbase = smem_u32(S.b[st]);
            // A slice p times the B slices 0 .. 6 - p goes to the groups p .. 6, whose accumulators lie
            // side by side: one product of up to 256 columns covers four of them
#pragma unroll
            for (int p = 0; p < kSlices; ++p) {
              const uint64_t ad = smem_desc(abase + p * (kTM * kTK * 2), kTM * 16, 128);
#pragma unroll
              for (int q = 0; q + p < kGroups; q += kWide) {
                const int w = kGroups - p - q < kWide ? kGroups - p - q : kWide;
                const uint64_t bd = smem_desc(bbase + q * (kTN * 16), kSlices * kTN * 16, 128);
                // the products of slice 0 in a chunk overwrite the accumulators
                mma_bf16(tmem + (uint32_t)((p + q) * kTN), ad, bd, instr_desc(w * kTN), (ks != kc || p > 0) ? 1u : 0u);
              }
            }
            mma_commit(&S.empty[st]);
            S.commits = u + 1;
          }
          mma_commit(&S.accf);  // tracks every MMA issued so far, whether or not an error stopped us
        }
      }
    }
  } else {
    // ---- fold and store
    const int q4 = warp & 3, cg = warp >> 2;  // TMEM lane quarter, group of 16 columns
    const uint32_t tcol = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(cg * 16);
    const int fe = fs - 63 - pexp;  // exponent of the fixed-point unit
    const long long f0 = FIXED && !base ? double_to_fixed(a0, fe) : 0;
    // 2^-39 and 2^-63 of the FP64 fold, times the table's exact scale 2^-pexp
    const double chi = FIXED ? 0.0 : ldexp(1.0, -39 - pexp), clo = FIXED ? 0.0 : ldexp(1.0, -63 - pexp);
    uint32_t chunk = 0;
    bool ok = true;
    for (int ti = 0; ti < my_tiles && ok; ++ti) {
      int tm, tn;
      coords((int)blockIdx.x + ti * (int)gridDim.x, tm, tn);
      const int t0 = tn * kTN + cg * 16;
      long long v[16];  // fixed-point sums, or the bits of FP64 sums
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = f0;
      for (int kc = 0; kc < nchunk; ++kc, ++chunk) {
        // (the whole warp leaves or stays: the tensor-memory loads below need it converged)
        if (__any_sync(0xffffffffu, S.err || !mbar_wait(&S.accf, chunk & 1))) {
          S.err = 1;
          ok = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          int ga[8];
          long long gb[8];
          {
            uint32_t r[4][8];
#pragma unroll
            for (int g = 0; g < 4; ++g) tmem_ld8_async(tcol + (uint32_t)(g * kTN + h * 8), r[g]);
#pragma unroll
            for (int g = 0; g < 4; ++g) tmem_wait(r[g]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              ga[i] = group_sum(r[0][i]) * 256 + group_sum(r[1][i]);
              gb[i] = (long long)group_sum(r[2][i]) * 256 + group_sum(r[3][i]);
            }
          }
          uint32_t r[3][8];
#pragma unroll
          for (int g = 0; g < 3; ++g) tmem_ld8_async(tcol + (uint32_t)((4 + g) * kTN + h * 8), r[g]);
#pragma unroll
          for (int g = 0; g < 3; ++g) tmem_wait(r[g]);
          if (h == 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.acce);  // the accumulators may be overwritten
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int s4 = group_sum(r[0][i]), s5 = group_sum(r[1][i]), s6 = group_sum(r[2][i]);
            long long& w = v[h * 8 + i];
            if (FIXED) {
              w = fold_fixed(ga[i], gb[i], s4, s5, s6, fs, w);
            } else {
              const long long hi = (long long)ga[i] * 65536 + gb[i], lo = (long long)s4 * 65536 + ((long long)s5 * 256 + s6);
              const double c = nchunk == 1 ? exact_fold(hi, lo, -63 - pexp)
                                           : __longlong_as_double(w) + fma((double)hi, chi, (double)lo * clo);
              w = __double_as_longlong(c);
            }
          }
        }
      }
      if (!ok) break;
      const int b = tm * kTM + q4 * 32 + lane;
      auto value = [&](int i) {
        if (FIXED) {
          long long z = v[i];
          if (base && t0 + i < nT) z = (long long)((unsigned long long)z + (unsigned long long)double_to_fixed(base[t0 + i], fe));
          return fixed_to_double(z, fe);
        }
        return (base ? (t0 + i < nT ? base[t0 + i] : 0.0) : a0) + __longlong_as_double(v[i]);
      };
      if (b < B) {
        double* o = out_row(O, nT, b, t0);
        if (t0 + 16 <= nT && ((uintptr_t)o & 31) == 0) {
#pragma unroll
          for (int i = 0; i < 16; i += 4) {
            const double d[4] = {value(i), value(i + 1), value(i + 2), value(i + 3)};
            st_sector(o + i, d);
          }
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (t0 + i < nT) o[i] = value(i);
        }
      }
      __syncwarp();
    }
  }
  __syncthreads();
  if (tid == 0) {
    if (S.err) {
      atomicOr(err_flag, 1);
      // drain the loads that no product consumed
      for (uint32_t u = S.uses; u < S.loads; ++u) mbar_wait(&S.full[u % kStages], (u / kStages) & 1);
    }
    // and the last products of every stage
    for (uint32_t u = S.commits > kStages ? S.commits - kStages : 0; u < S.commits; ++u)
      mbar_wait(&S.empty[u % kStages], (u / kStages) & 1);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

int grid1(size_t n) {
  size_t g = (n + 255) / 256;
  return (int)(g < 1 ? 1 : (g > 152 * 64 ? 152 * 64 : g));
}

// cuTensorMapEncodeTiled through the runtime's driver entry points (no link-time dependency)
typedef CUresult (*EncodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encoder() {
  static std::once_flag once;
  static EncodeTiled fn = nullptr;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiled)f;
  });
  return fn;
}

// tensor map of slices [7][kpad/8][rows_pad][8] (BF16), one K step of all slices per box: 8 x box_rows x
// 2 x 7, or, with the slices of one K half side by side, 8 x box_rows x 7 x 2
cudaError_t slice_map(CUtensorMap* m, const void* base, int rows_pad, int kpad, int box_rows, bool slices_inner) {
  EncodeTiled enc = encoder();
  if (!enc) return cudaErrorNotSupported;
  const int ks = slices_inner ? 3 : 2, sl = slices_inner ? 2 : 3;  // dimensions of K halves and of slices
  cuuint64_t dim[4] = {8, (cuuint64_t)rows_pad, 0, 0}, stride[3] = {16, 0, 0};
  cuuint32_t box[4] = {8, (cuuint32_t)box_rows, 0, 0};
  dim[ks] = (cuuint64_t)(kpad / 8), stride[ks - 1] = (cuuint64_t)rows_pad * 16, box[ks] = 2;
  dim[sl] = (cuuint64_t)kSlices, stride[sl - 1] = stride[ks - 1] * (cuuint64_t)(kpad / 8), box[sl] = (cuuint32_t)kSlices;
  const cuuint32_t es[4] = {1, 1, 1, 1};
  const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dim, stride, box, es,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

size_t tc_slices_bytes(int rows, int k) {
  const size_t rp = ((size_t)rows + 127) / 128 * 128, kp = ((size_t)k + 15) / 16 * 16;
  return (size_t)kSlices * rp * kp * sizeof(__nv_bfloat16);
}

int tc_pad_rows(int rows) { return (rows + 127) / 128 * 128; }
int tc_pad_k(int k) { return (k + 15) / 16 * 16; }

cudaError_t launch_psi_slices(const double* d_psi, int s_rows, int nT, void* d_out, cudaStream_t st, int pexp) {
  // psi is [s_rows][nT] (row = term j): the slices are [7][K_pad/8][nT_pad][8] of 2^pexp psi
  const int rp = tc_pad_rows(nT), kp = tc_pad_k(s_rows);
  k_slice_rows<<<grid1((size_t)rp * kp), 256, 0, st>>>(d_psi, nT, s_rows, 1, (size_t)nT, std::ldexp(128.0, pexp), rp,
                                                      kp, (__nv_bfloat16*)d_out);
  return cudaGetLastError();
}

cudaError_t launch_y_slices(const double* d_Y, int B, int ldy, int k, int kpad, void* d_out, cudaStream_t st) {
  const int rp = tc_pad_rows(B);
  k_slice_rows<<<grid1((size_t)rp * kpad), 256, 0, st>>>(d_Y, B, k, (size_t)ldy, 1, 256.0, rp, kpad,
                                                        (__nv_bfloat16*)d_out);
  return cudaGetLastError();
}

// a[B][nT] = a0 + Y psi from slices: y slices [7][kpad/8][Bpad][8] built for K = kpad columns, psi
// slices [7][kpad_psi/8][nTpad][8] (only the first kpad columns are read)
namespace {
cudaError_t coef_tc(const void* d_yslices, int B, int kpad, const void* d_pslices, int nT, int kpad_psi, double a0,
                    const TcOut& O, int* d_err, cudaStream_t st, const double* d_base, int pexp, double amax) {
  if (B == 0 || nT == 0) return cudaSuccess;
  if (kpad > kpad_psi || kpad % kTK || kpad <= 0) return cudaErrorInvalidValue;
  const int Bp = tc_pad_rows(B), nTp = tc_pad_rows(nT);
  // the fixed-point unit: the smallest fs >= 1 with |a| < 2^{fs - pexp} (see k_coef_tc)
  int fs = 1;
  while (fs <= 8 && !(std::ldexp(amax, pexp) < std::ldexp(1.0, fs))) ++fs;
  // a zeroth term far below the terms has to be a multiple of that unit too, as it is from 2^{fs - 11 - pexp} on
  const bool fixed = fs <= 8 && (d_base || a0 >= std::ldexp(1.0, fs - 11 - pexp));
  const int T = kpad / kTK;
  // sample slices of a row tile kept in shared memory: up to kResSteps K steps, in fixed point (the others need
  // the larger stages, respectively the registers, of k_coef_tc).  Measured at K = 64, mesh 1/64, 2,048
  // samples: 115 us streamed, 80 us resident.
  const bool resident = fixed && T <= kResSteps;
  CUtensorMap tmY, tmP;
  cudaError_t e = slice_map(&tmY, d_yslices, Bp, kpad, kTM, false);
  if (e != cudaSuccess) return e;
  // the psi slices hold kpad_psi columns; the map covers them all, the kernel reads kpad
  e = slice_map(&tmP, d_pslices, nTp, kpad_psi, resident ? kRN : kTN, true);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const int ntm = Bp / kTM, ntn = (nT + (resident ? kRN : kTN) - 1) / (resident ? kRN : kTN);
  const long ntiles = (long)ntm * ntn;
  if (ntiles > 0x7fffffffL) return cudaErrorInvalidValue;
  const int grid = (int)(ntiles < sms ? ntiles : sms);
  // shared memory limits are raised once per device (never lowered), so the launch can also be captured
  if (resident) {
    const int nst = std::min(kResStages, (int)((kResSmem - T * kABytes) / (T * kRBytes)));
    const size_t smem = (size_t)T * kABytes + (size_t)nst * T * kRBytes + 1024;
    const auto kern = T <= 2   ? k_coef_res<small_groups(2)>
                      : T == 3 ? k_coef_res<small_groups(3)>
                      : T == 4 ? k_coef_res<small_groups(4)>
                               : k_coef_res<small_groups(5)>;
    if ((e = raise_smem_limit((const void*)kern, kResSmem + 1024)) != cudaSuccess) return e;
    kern<<<grid, kTcThreads, smem, st>>>(tmY, tmP, B, nT, T, nst, ntn, (int)ntiles, a0, O, d_err, d_base, pexp, fs);
    return cudaGetLastError();
  }
  const size_t smem = sizeof(TcSmem) + 1024;
  const void* kern = fixed ? (const void*)k_coef_tc<true> : (const void*)k_coef_tc<false>;
  if ((e = raise_smem_limit(kern, (int)smem)) != cudaSuccess) return e;
  if (fixed)
    k_coef_tc<true><<<grid, kTcThreads, smem, st>>>(tmY, tmP, B, nT, kpad, ntm, (int)ntiles, a0, O, d_err, d_base, pexp, fs);
  else
    k_coef_tc<false><<<grid, kTcThreads, smem, st>>>(tmY, tmP, B, nT, kpad, ntm, (int)ntiles, a0, O, d_err, d_base, pexp, 0);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_coef_tc(const void* d_yslices, int B, int kpad, const void* d_pslices, int nT, int kpad_psi,
                           double a0, double* d_a, int* d_err, cudaStream_t st, const double* d_base, int pexp,
                           double amax) {
  const TcOut O{d_a, 0, 0, 0, 0};
  return coef_tc(d_yslices, B, kpad, d_pslices, nT, kpad_psi, a0, O, d_err, st, d_base, pexp, amax);
}

size_t sep_tables_bytes(int n, int k1pad, int k2max) {
  return 2 * tc_slices_bytes(n, k1pad) + (size_t)(k2max + 1) * n * sizeof(int2) + 4 * 256;
}

cudaError_t launch_sep_tables(int n, int k1max, int k1pad, int k2max, double* d_work, void* d_tables, SepTables* t,
                              cudaStream_t st) {
  char* p = (char*)d_tables;
  auto take = [&](size_t bytes) {
    p = (char*)(((uintptr_t)p + 255) & ~(uintptr_t)255);
    char* r = p;
    p += bytes;
    return r;
  };
  t->k1pad = k1pad;
  t->sy = (int2*)take((size_t)(k2max + 1) * n * sizeof(int2));
  k_sep_sy<<<grid1((size_t)(k2max + 1) * n), 256, 0, st>>>(n, k2max, (int2*)t->sy);
  for (int plane = 0; plane < 2; ++plane) {
    t->sx[plane] = take(tc_slices_bytes(n, k1pad));
    k_sep_sx<<<grid1((size_t)n * k1pad), 256, 0, st>>>(n, plane, k1max, k1pad, d_work);
    const int rp = tc_pad_rows(n);
    k_slice_rows<<<grid1((size_t)rp * k1pad), 256, 0, st>>>(d_work, n, k1pad, (size_t)k1pad, 1, 128.0, rp, k1pad,
                                                           (__nv_bfloat16*)t->sx[plane]);
  }
  return cudaGetLastError();
}

// the slices of one plane in the scratch
static size_t sep_plane_bytes(int B, int n, int k1pad) { return (tc_slices_bytes(B * n, k1pad) + 255) & ~(size_t)255; }

size_t sep_scratch_bytes(int B, int n, int nlist, int k1pad) {
  return 2 * sep_plane_bytes(B, n, k1pad) + (size_t)B * nlist * sizeof(int2) + (size_t)2 * k1pad * sizeof(int);
}

cudaError_t launch_coef_sep(const double* d_Y, int ldy, int B, int K, int k1pad, const SepTerms& terms,
                            const SepTables& tab, int n, double a0, int ey, void* d_tslices, double* d_a, int* d_err,
                            cudaStream_t st, double amax) {
  if (B == 0) return cudaSuccess;
  if (k1pad % kTK || k1pad <= 0 || k1pad > tab.k1pad || (long)B * n > 0x7fffffffL - 128) return cudaErrorInvalidValue;
  const int rows = B * n, rp = tc_pad_rows(rows);
  const size_t pb = sep_plane_bytes(B, n, k1pad);
  int2* yc = (int2*)((char*)d_tslices + 2 * pb);
  int* kend = (int*)(yc + (size_t)B * terms.nlist);
  __nv_bfloat16* const sl[2] = {(__nv_bfloat16*)d_tslices, (__nv_bfloat16*)((char*)d_tslices + pb)};
  k_sep_yc<<<grid1((size_t)std::max(B * (long)terms.nlist, 2L * k1pad)), 256, 0, st>>>(
      d_Y, ldy, B, K, terms.cj, terms.list, terms.start, terms.nlist, 2 * k1pad, std::ldexp(1.0, 60 + ey), yc, kend);
  k_sep_stage1<<<grid1((size_t)rp * (k1pad / 8)), 256, 0, st>>>(yc, B, n, terms.nlist, k1pad, terms.start, kend, terms.list,
                                                               tab.sy, rp, sl[0], sl[1]);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  for (int plane = 0; plane < 2; ++plane) {
    // rows (b, j) of this plane land at a[b][plane][j][.]: b 2n^2 + plane n^2 + j n
    const TcOut O{d_a + (size_t)plane * n * n, n, 2LL * n * n, (long long)n, 1};
    if ((e = coef_tc(sl[plane], rows, k1pad, tab.sx[plane], n, tab.k1pad, a0, O, d_err, st, nullptr, ey, amax)) !=
        cudaSuccess)
      return e;
  }
  return cudaSuccess;
}

}  // namespace mq

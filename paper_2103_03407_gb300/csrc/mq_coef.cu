// Lattice points and centroid coefficients (the data-parallel front of the level evaluation).
//
//  * lattice_points: y = {k z / N + Delta_r} - 1/2 (Sec. 2.5, eq. rqmc; eq. t_kl), exact integer
//    arithmetic for k z mod N, one IEEE division and the same wrap as the fractional part.
//  * psi_table: Psi[j][t] = c_j sin(pi k1_j x_t) sin(pi k2_j y_t) at the centroids of the
//    2 n^2 triangles (lower triangle of cell (i,j): ((3i+2)/(3n), (3j+1)/(3n)); upper:
//    ((3i+1)/(3n), (3j+2)/(3n))), optionally restricted to the islands D_f of the second test
//    problem of Sec. 5 or to their complement (region code per term).
//  * island_field: the piecewise-constant zeroth terms a_0, b_0 of that problem.
//  * coef_gemm_f64: a[b][t] = a0 + sum_{j<s} Y[b][j] Psi[j][t] (eq. coeff, eq. coeff_s) as a
//    tiled FP64 GEMM (register-blocked 4 x 8 outputs per thread, shared-memory K tiles); with a
//    base field, base[t] in place of the constant a0.
#include <cuda_runtime.h>

#include <cstdint>

#include "mq_internal.h"

namespace mq {
namespace {

// mbits > 0: the embedded rule of 2^mbits points in radical-inverse order, point k taking the
// lattice index rev(k) (the mbits-bit reversal of k) with N = 2^mbits, so the first 2^m points are
// the 2^m-point rule (Sec. 2.5, embedded lattice rules)
// dk: NULL, or a device offset added to k0 (a captured graph replayed on another range)
__global__ void lattice_kernel(const uint32_t* __restrict__ z, uint32_t N, const double* __restrict__ delta, int R,
                               int s, uint32_t k0, int npts, int mbits, const uint32_t* dk, double* __restrict__ Y) {
  if (dk) k0 += *dk;
  const size_t tot = (size_t)R * npts * s;
  for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < tot; q += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(q % s);
    const size_t b = q / s;
    const int kk = (int)(b % npts);
    const int r = (int)(b / npts);
    uint64_t k = (uint64_t)k0 + (uint64_t)kk;
    if (mbits > 0) k = (uint64_t)(__brev((uint32_t)k) >> (32 - mbits));
    const uint64_t m = (k * (uint64_t)z[j]) % (uint64_t)N;
    double t = (double)m / (double)N + delta[(size_t)r * s + j];
    if (t >= 1.0) t -= 1.0;
    Y[q] = t - 0.5;
  }
}

// Whether the centroid num / (3n) (one coordinate) lies in [1/8, 3/8] or [5/8, 7/8], decided in
// integers: 8 num against 3n, 9n, 15n, 21n.  (A centroid never lies on such a line: 8 num is not a
// multiple of 3, 3 n m is.)
__device__ __forceinline__ bool island_band(long num, long n) {
  const long e = 8 * num;
  return (e >= 3 * n && e <= 9 * n) || (e >= 15 * n && e <= 21 * n);
}

// numerators of the centroid of triangle t (plane 0: lower, 1: upper) of cell (i, j) over 3n
__device__ __forceinline__ void centroid_num(int n, size_t t, long& nx, long& ny) {
  const size_t nn = (size_t)n * n;
  const int plane = (int)(t / nn);
  const size_t cell = t % nn;
  const int i = (int)(cell % n), jj = (int)(cell / n);
  nx = 3L * i + (plane == 0 ? 2 : 1);
  ny = 3L * jj + (plane == 0 ? 1 : 2);
}

__global__ void psi_kernel(int n, int s, const int* __restrict__ k1, const int* __restrict__ k2,
                           const double* __restrict__ cj, const int* __restrict__ region, double* __restrict__ psi) {
  const size_t nn = (size_t)n * n, nT = 2 * nn, tot = (size_t)s * nT;
  for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < tot; q += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(q / nT);
    const size_t t = q % nT;
    long nx, ny;
    centroid_num(n, t, nx, ny);
    // k x modulo 2 in integers (x = nx / 3n): the argument keeps FP64 accuracy however large k is
    const double x = (double)((k1[j] * nx) % (6L * n)) / (double)(3 * n);
    const double y = (double)((k2[j] * ny) % (6L * n)) / (double)(3 * n);
    double v = cj[j] * sinpi(x) * sinpi(y);
    if (region && region[j]) {
      const bool in = island_band(nx, n) && island_band(ny, n);
      if (in != (region[j] == 1)) v = 0.0;
    }
    psi[q] = v;
  }
}

__global__ void island_kernel(int n, double v_in, double v_out, double* __restrict__ base) {
  const size_t nT = (size_t)2 * n * n;
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < nT; t += (size_t)gridDim.x * blockDim.x) {
    long nx, ny;
    centroid_num(n, t, nx, ny);
    base[t] = (island_band(nx, n) && island_band(ny, n)) ? v_in : v_out;
  }
}

// FP64 fused multiply-add throughput: eight independent chains per thread keep the FP64 pipes
// busy (the denominator of the per-sample kernel's FP64 roofline)
__global__ void __launch_bounds__(256) fp64_fma_kernel(double* out, int iters, double a, double b) {
  double x[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) x[i] = 1e-3 * threadIdx.x + i;
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = fma(x[i], a, b);
  }
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < 8; ++i) s += x[i];
  if (s == -1.0) out[0] = s;  // never true; keeps the chains alive
}

constexpr int GBM = 64, GBN = 128, GBK = 16;

// C[b][t] = a0 + sum_j Y[b*ldy + j] Psi[j*nT + t]; 256 threads as 16 x 16, 4 x 8 outputs each.
__global__ void __launch_bounds__(256) gemm_f64_kernel(const double* __restrict__ Y, int ldy, int B, int s,
                                                       const double* __restrict__ Psi, int nT, double a0,
                                                       double* __restrict__ C, const double* __restrict__ base) {
  __shared__ double As[GBK][GBM + 1];
  __shared__ double Bs[GBK][GBN];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int b0 = blockIdx.y * GBM, t0 = blockIdx.x * GBN;
  double acc[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.0;
  for (int k0 = 0; k0 < s; k0 += GBK) {
    // Y tile: 64 rows x 16 k
    for (int q = threadIdx.x; q < GBM * GBK; q += 256) {
      const int rr = q / GBK, kk = q % GBK;
      const int b = b0 + rr, k = k0 + kk;
      As[kk][rr] = (b < B && k < s) ? Y[(size_t)b * ldy + k] : 0.0;
    }
    // Psi tile: 16 k x 128 t
    for (int q = threadIdx.x; q < GBK * GBN; q += 256) {
      const int kk = q / GBN, cc = q % GBN;
      const int k = k0 + kk, t = t0 + cc;
      Bs[kk][cc] = (k < s && t < nT) ? Psi[(size_t)k * nT + t] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < GBK; ++kk) {
      double a[4], bv[8];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 8; ++j) bv[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fma(a[i], bv[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int b = b0 + ty + 16 * i;
    if (b >= B) continue;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int t = t0 + tx + 16 * j;
      if (t < nT) C[(size_t)b * nT + t] = (base ? base[t] : a0) + acc[i][j];
    }
  }
}

int grid_for(size_t tot, int threads) {
  size_t g = (tot + threads - 1) / threads;
  if (g > 152 * 32) g = 152 * 32;
  if (g < 1) g = 1;
  return (int)g;
}

}  // namespace

cudaError_t measure_fp64_peak(int device, double* tflops, double* ms_out) {
  cudaError_t e = cudaSetDevice(device);
  if (e != cudaSuccess) return e;
  int sms = 0;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device)) != cudaSuccess) return e;
  double* d = nullptr;
  if ((e = cudaMalloc(&d, sizeof(double))) != cudaSuccess) return e;
  cudaStream_t st = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  const int blocks = sms * 8, threads = 256, iters = 1 << 14;
  float best = 1e30f;
  for (int rep = 0; rep < 4 && e == cudaSuccess; ++rep) {
    cudaEventRecord(e0, st);
    fp64_fma_kernel<<<blocks, threads, 0, st>>>(d, iters, 0.9999999, 1e-7);
    cudaEventRecord(e1, st);
    if ((e = cudaEventSynchronize(e1)) != cudaSuccess) break;
    float t = 0.0f;
    cudaEventElapsedTime(&t, e0, e1);
    if (rep > 0 && t < best) best = t;  // the first launch warms up
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (st) cudaStreamDestroy(st);
  cudaFree(d);
  if (e != cudaSuccess) return e;
  const double flops = 2.0 * 8.0 * iters * (double)blocks * threads;
  *tflops = flops / (best * 1e-3) / 1e12;
  *ms_out = best;
  return cudaSuccess;
}

cudaError_t launch_lattice_points(const uint32_t* d_z, uint32_t N, const double* d_delta, int R, int s, uint32_t k0,
                                  int npts, int mbits, double* d_Y, cudaStream_t st, const uint32_t* d_kshift) {
  const size_t tot = (size_t)R * npts * s;
  if (tot == 0) return cudaSuccess;
  if (mbits < 0 || mbits > 31 || (mbits > 0 && N != (1u << mbits))) return cudaErrorInvalidValue;
  lattice_kernel<<<grid_for(tot, 256), 256, 0, st>>>(d_z, N, d_delta, R, s, k0, npts, mbits, d_kshift, d_Y);
  return cudaGetLastError();
}

cudaError_t launch_psi_table(int n, int s, const int* d_k1, const int* d_k2, const double* d_cj, double* d_psi,
                             cudaStream_t st, const int* d_region) {
  const size_t tot = (size_t)s * 2 * n * n;
  if (tot == 0) return cudaSuccess;
  psi_kernel<<<grid_for(tot, 256), 256, 0, st>>>(n, s, d_k1, d_k2, d_cj, d_region, d_psi);
  return cudaGetLastError();
}

cudaError_t launch_island_field(int n, double v_in, double v_out, double* d_base, cudaStream_t st) {
  const size_t tot = (size_t)2 * n * n;
  island_kernel<<<grid_for(tot, 256), 256, 0, st>>>(n, v_in, v_out, d_base);
  return cudaGetLastError();
}

cudaError_t launch_coef_gemm_f64(const double* d_Y, int ldy, int B, int s, const double* d_psi, int nT, double a0,
                                 double* d_a, cudaStream_t st, const double* d_base) {
  if (B == 0 || nT == 0) return cudaSuccess;
  dim3 grid((nT + GBN - 1) / GBN, (B + GBM - 1) / GBM);
  if (grid.y > 65535) return cudaErrorInvalidValue;
  gemm_f64_kernel<<<grid, 256, 0, st>>>(d_Y, ldy, B, s, d_psi, nT, a0, d_a, d_base);
  return cudaGetLastError();
}

}  // namespace mq

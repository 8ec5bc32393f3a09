// Per-sample two-grid kernel: one CTA evaluates whole samples of one MLQMC level.
//
// For each sample (shift r, lattice point k) the CTA
//   1. builds the coarse-mesh operator from the centroid coefficients (truncation S_l) and
//      computes the smallest eigenpair (lambda_H, u_H) by LOBPCG preconditioned with a
//      multigrid V-cycle, warm-started from the eigenvector of the previous lattice point of
//      its chain (Sec. 4.3, "reusing samples from nearby QMC points");
//   2. for the fine mesh of the level (and, on l > 0, the fine mesh of level l-1, from the same
//      coarse pair -- Algorithm 2), forms b = M_h P u_H (P: P1 interpolation), solves
//      (A_h - lambda_H M_h) w = b (eq. 2grid_source) by MINRES preconditioned with a symmetric
//      multigrid V-cycle on A_h, inside iterative refinement (solution, right-hand side and residual in
//      FP64, in the FP32 kernel as double-floats: pairs of FP32, 48 bits), and returns the Rayleigh
//      quotient w^T A_h w / w^T M_h w (Algorithm 1 steps 3-4, eq. RQ_update);
//   3. writes lambda_H, lambda^l, lambda^{l-1} and the difference (or, for the functional
//      quantity of interest, lambda_H and G of the two eigenfunction approximations and their
//      difference, G(u) = |integral of u| / ||u||_L2).
//
// With a reaction term (the second test problem of Sec. 5) every operator above is A + B, B the
// reaction matrix of b (seven-point form, see mq_device.cuh), and the V-cycles precondition with
// A + D_B (the lumped reaction).
//
// Operators are matrix-free.  On the SW-NE triangulation with centroid coefficients the P1
// stiffness is the weighted five-point edge form
//     (A x)_p = sum_{edges pq} w_pq (x_p - x_q),
//     w of edge (i,j)-(i+1,j) = (a_low(i,j) + a_up(i,j-1)) / 2,
//     w of edge (i,j)-(i,j+1) = (a_up(i,j) + a_low(i-1,j)) / 2
// (the hypotenuses carry no weight), and the consistent mass is the seven-point form
//     (M x)_p = h^2/12 (6 x_p + x_E + x_W + x_N + x_S + x_NE + x_SW).
// Vectors live on the padded (n+1) x (n+1) node grid with a zero boundary ring, so every
// stencil is branch-free.  The multigrid coarse operators are the Galerkin operators P^T A P,
// which for nested P1 spaces are the coarse P1 stiffness with each coarse triangle's
// coefficient the mean of its four fine triangles.
//
// Workspace: one slab per CTA, carved identically on host (to size it) and device.  The slab
// lives in dynamic shared memory when it fits, otherwise in a global scratch buffer.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <map>
#include <mutex>
#include <utility>

#include "mq_device.cuh"
#include "mq_internal.h"

namespace mq {
namespace {

using namespace dev;

// Coarse eigensolve workspace: FP64 LOBPCG basis, FP64 operator weights, FP32 preconditioner.
struct CoarseWS {
  MGDesc<float> mg;
  double *wx, *wy;
  double *rx, *ry, *rd;  // reaction edge weights (NULL without a reaction term)
  double *x, *Ax, *Mx, *w, *Aw, *Mw, *p, *Ap, *Mp, *uprev;
  float *r32, *w32;
};

// uprev comes first: it holds the coarse eigenvector through the fine solves (and as the warm
// start of the next point), while the rest of the coarse workspace is dead during the fine solves
// and shares its memory with the fine workspace.  *persist receives the bytes of that head.
__host__ __device__ void carve_coarse(Carver& c, int nc, CoarseWS& ws, size_t* persist = nullptr,
                                      bool reaction = false) {
  const size_t V = gsz(nc);
  ws.uprev = c.take<double>(V);
  if (persist) *persist = c.used();
  ws.wx = c.take<double>(V);
  ws.wy = c.take<double>(V);
  ws.rx = reaction ? c.take<double>(V) : nullptr;
  ws.ry = reaction ? c.take<double>(V) : nullptr;
  ws.rd = reaction ? c.take<double>(V) : nullptr;
  ws.x = c.take<double>(V);
  ws.Ax = c.take<double>(V);
  ws.Mx = c.take<double>(V);
  ws.w = c.take<double>(V);
  ws.Aw = c.take<double>(V);
  ws.Mw = c.take<double>(V);
  ws.p = c.take<double>(V);
  ws.Ap = c.take<double>(V);
  ws.Mp = c.take<double>(V);
  ws.r32 = c.take<float>(V);
  ws.w32 = c.take<float>(V);
  carve_mg<float>(c, nc, ws.mg, reaction);
}

// Coarse eigensolve workspace of the FP32 kernel (lobpcg32): the iterate as a double-float pair, the
// operator's weights as pairs (their high parts are the multigrid hierarchy's finest weights), the
// search directions and their images in FP32.
struct CoarseWS32 {
  MGDesc<float> mg;
  float *xh, *xl, *wxl, *wyl, *r, *w, *mw, *p, *ap, *mp;
  float *rx, *ry, *rd, *rxl, *ryl, *rdl;  // reaction edge weights and their low parts (NULL without a reaction term)
};

// Meshes up to which the FP32 kernel takes its own form of a solve on the coarse mesh itself (`near` below)
constexpr int kNear32Max = 128;

// xh, xl come first: they hold the coarse eigenvector through the fine solves
__host__ __device__ void carve_coarse32(Carver& c, int nc, CoarseWS32& ws, size_t* persist = nullptr,
                                        bool reaction = false) {
  const size_t V = gsz(nc);
  ws.xh = c.take<float>(V);
  ws.xl = c.take<float>(V);
  if (persist) *persist = c.used();
  float** const a[8] = {&ws.wxl, &ws.wyl, &ws.r, &ws.w, &ws.mw, &ws.p, &ws.ap, &ws.mp};
  for (float** v : a) *v = c.take<float>(V);
  float** const b[6] = {&ws.rx, &ws.ry, &ws.rd, &ws.rxl, &ws.ryl, &ws.rdl};
  for (float** v : b) *v = reaction ? c.take<float>(V) : nullptr;
  carve_mg<float>(c, nc, ws.mg, reaction, false);
  // the coefficients of the coarser meshes are needed only while the hierarchy is built, before ap and mp are
  ws.mg.cell[0] = ws.ap;
  ws.mg.cell[1] = ws.mp;
  ws.mg.rcell[0] = reaction ? ws.mw : nullptr;
  ws.mg.rcell[1] = reaction ? c.take<float>((size_t)nc * nc / 2 + 1) : nullptr;
}

// Fine shifted-solve workspace: solution and right-hand side beyond FP32, inner vectors in T.  Its size sets how many
// blocks share an SM, and the kernel is bound by the latency of its phases: without arrays of their own for q, the
// inner solution and the coarse coefficients, mesh 1/16 takes 22.8 instead of 26.1 KB (FP64: 34.8 / 41.7 KB), eight
// blocks per SM instead of seven (five / four).  8,192 samples of the first test problem's level 1: 8.2 -> 7.7
// ms, 2,048 samples of the smallest FP64 workload: 2.48 -> 2.33 ms.
template <typename T>
struct FineWS {
  MGDesc<T> mg;
  double *x64, *b64;  // FP64 kernel
  // FP32 kernel: solution and right-hand side as double-floats, the low parts of the edge weights (and of
  // the reaction's)
  float *xh, *xl, *bh, *bl, *wxl, *wyl, *rxl, *ryl, *rdl;
  T *vo, *v, *z, *zn, *wo, *w;
  T *rx, *ry, *rd;  // reaction edge weights in the inner precision (NULL without a reaction term)
};

template <typename T>
__host__ __device__ void carve_fine(Carver& c, int n, FineWS<T>& ws, bool reaction = false) {
  const size_t V = gsz(n);
  const bool f32 = sizeof(T) == sizeof(float);
  ws.x64 = f32 ? nullptr : c.take<double>(V);
  ws.b64 = f32 ? nullptr : c.take<double>(V);
  float** const pr[6] = {&ws.xh, &ws.xl, &ws.bh, &ws.bl, &ws.wxl, &ws.wyl};
  for (float** v : pr) *v = f32 ? c.take<float>(V) : nullptr;
  float** const rl[3] = {&ws.rxl, &ws.ryl, &ws.rdl};
  for (float** v : rl) *v = f32 && reaction ? c.take<float>(V) : nullptr;
  ws.vo = c.take<T>(V);
  ws.v = c.take<T>(V);
  ws.z = c.take<T>(V);
  ws.zn = c.take<T>(V);
  ws.wo = c.take<T>(V);
  ws.w = c.take<T>(V);
  ws.rx = reaction ? c.take<T>(V) : nullptr;
  ws.ry = reaction ? c.take<T>(V) : nullptr;
  ws.rd = reaction ? c.take<T>(V) : nullptr;
  carve_mg<T>(c, n, ws.mg, reaction, false);
  // the coefficients of the coarser meshes are needed only while the hierarchy is built; of wo and w only
  // interiors are read, after they have been written
  ws.mg.cell[0] = ws.wo;
  ws.mg.cell[1] = ws.w;
  const size_t cells = n >= 4 ? (size_t)2 * (n / 2) * (n / 2) : 1;
  for (int k = 0; k < 2; ++k) ws.mg.rcell[k] = reaction ? c.take<T>(cells) : nullptr;
}

template <typename T>
__host__ __device__ size_t fine_bytes(int n, bool reaction = false) {
  if (n < 2) return 0;
  Carver f(nullptr);
  FineWS<T> fw;
  carve_fine<T>(f, n, fw, reaction);
  return (f.used() + 15) & ~(size_t)15;
}

// workspace of one CTA: the persistent head, then the larger of the rest of the coarse region
// and the largest fine solve it performs in place (mode 2: not in this kernel).  A multiple of 256 bytes: the slabs of a global scratch lie back
// to back, so every slab then starts as aligned as the scratch itself and the kernel carves it
// exactly as sized here (an unaligned slab start would shift its arrays by up to 15 bytes into
// the next slab).
template <typename T>
__host__ __device__ size_t slab_size(int nf, int nc, int np, bool eig32, int mode_f, int mode_p, bool reaction) {
  Carver c(nullptr);
  size_t persist = 0;
  if (sizeof(T) == sizeof(float) && eig32) {
    CoarseWS32 cw;
    carve_coarse32(c, nc, cw, &persist, reaction);
  } else {
    CoarseWS cw;
    carve_coarse(c, nc, cw, &persist, reaction);
  }
  persist = (persist + 15) & ~(size_t)15;  // the fine region starts 16-byte aligned
  const size_t coarse = (c.used() + 15) & ~(size_t)15;
  auto need = [&](int n, int mode) -> size_t {
    // (the FP32 kernel's FP64 solve on a large coarse mesh itself has its own workspace)
    if (mode == 2 || (sizeof(T) == sizeof(float) && n == nc && nc > kNear32Max)) return 0;
    return fine_bytes<T>(n, reaction);
  };
  size_t m = coarse - persist;
  const size_t a = need(nf, mode_f), b = need(np, mode_p);
  if (a > m) m = a;
  if (b > m) m = b;
  return (persist + m + 255) & ~(size_t)255;
}

// ---------------------------------------------------------------------------------------------
// Small dense Rayleigh-Ritz for LOBPCG, run by one thread.  The pencil is shifted by the current
// Ritz value in FP64 before it is rounded to FP32: the shifted Gram matrix GA - theta GM has
// entries of the size of the correction, so FP32 resolves the correction to FP32 relative
// accuracy (GB300 executes FP64 at a small fraction of the FP32 rate, and a single thread's FP64
// instruction costs a full warp's issue slot).  Basis [x, w, p] (k = 2 or 3).  Returns the number
// of basis vectors kept (0: failure), the coefficients c of the smallest Ritz vector and mu, the
// smallest eigenvalue of the shifted pencil (theta_new - theta).
__device__ int rayleigh_ritz_shifted(const float GAs[3][3], const float GM[3][3], int k, float c[3], float& mu) {
  for (; k >= 2; --k) {
    float dsc[3], A[3][3], B[3][3], Lm[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    bool ok = true;
    for (int i = 0; i < k; ++i) {
      if (!(GM[i][i] > 0.0f)) ok = false;
      dsc[i] = ok ? rsqrtf(GM[i][i]) : 0.0f;
    }
    if (!ok) continue;
    for (int i = 0; i < k; ++i)
      for (int j = 0; j < k; ++j) {
        A[i][j] = dsc[i] * GAs[i][j] * dsc[j];
        B[i][j] = dsc[i] * GM[i][j] * dsc[j];
      }
    for (int i = 0; i < k && ok; ++i)
      for (int j = 0; j <= i; ++j) {
        float s = B[i][j];
        for (int m = 0; m < j; ++m) s -= Lm[i][m] * Lm[j][m];
        if (i == j) {
          if (!(s > 1e-5f)) {
            ok = false;
            break;
          }
          Lm[i][i] = sqrtf(s);
        } else {
          Lm[i][j] = s / Lm[j][j];
        }
      }
    if (!ok) continue;
    float Y[3][3], C[3][3];
    for (int j = 0; j < k; ++j)
      for (int i = 0; i < k; ++i) {
        float s = A[i][j];
        for (int m = 0; m < i; ++m) s -= Lm[i][m] * Y[m][j];
        Y[i][j] = s / Lm[i][i];
      }
    for (int i = 0; i < k; ++i)
      for (int j = 0; j < k; ++j) {
        float s = Y[i][j];
        for (int m = 0; m < j; ++m) s -= Lm[j][m] * C[i][m];
        C[i][j] = s / Lm[j][j];
      }
    for (int i = 0; i < k; ++i)
      for (int j = 0; j < i; ++j) C[i][j] = C[j][i] = 0.5f * (C[i][j] + C[j][i]);
    float V[3][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}};
    for (int sweep = 0; sweep < 12; ++sweep) {
      float off = 0.0f, dia = 0.0f;
      for (int i = 0; i < k; ++i) {
        dia += C[i][i] * C[i][i];
        for (int j = i + 1; j < k; ++j) off += C[i][j] * C[i][j];
      }
      if (off <= 1e-14f * dia || off == 0.0f) break;
      for (int pI = 0; pI < k - 1; ++pI)
        for (int qI = pI + 1; qI < k; ++qI) {
          const float apq = C[pI][qI];
          if (apq == 0.0f) continue;
          const float tau = (C[qI][qI] - C[pI][pI]) / (2.0f * apq);
          const float t = (tau >= 0 ? 1.0f : -1.0f) / (fabsf(tau) + sqrtf(1.0f + tau * tau));
          const float cs = rsqrtf(1.0f + t * t), sn = t * cs;
          for (int m = 0; m < k; ++m) {
            const float cmp = C[m][pI], cmq = C[m][qI];
            C[m][pI] = cs * cmp - sn * cmq;
            C[m][qI] = sn * cmp + cs * cmq;
          }
          for (int m = 0; m < k; ++m) {
            const float cpm = C[pI][m], cqm = C[qI][m];
            C[pI][m] = cs * cpm - sn * cqm;
            C[qI][m] = sn * cpm + cs * cqm;
          }
          for (int m = 0; m < k; ++m) {
            const float vmp = V[m][pI], vmq = V[m][qI];
            V[m][pI] = cs * vmp - sn * vmq;
            V[m][qI] = sn * vmp + cs * vmq;
          }
        }
    }
    int mi = 0;
    for (int i = 1; i < k; ++i)
      if (C[i][i] < C[mi][mi]) mi = i;
    mu = C[mi][mi];
    float y[3] = {V[0][mi], V[1][mi], k > 2 ? V[2][mi] : 0.0f};
    float cc[3] = {0, 0, 0};
    for (int i = k - 1; i >= 0; --i) {
      float s = y[i];
      for (int m = i + 1; m < k; ++m) s -= Lm[m][i] * cc[m];
      cc[i] = s / Lm[i][i];
    }
    for (int i = 0; i < 3; ++i) c[i] = i < k ? cc[i] * dsc[i] : 0.0f;
    return k;
  }
  return 0;
}

struct EigShared {
  double c[3];   // x_new = c0 x + c1 w + c2 p
  double pc[2];  // p_new = pc0 w + pc1 p
  double theta;
  double scale;  // normalisation factor
  int k;
  int conv;
};

// LOBPCG for the smallest eigenpair of (A_H, M_H), preconditioned by one FP32 V-cycle on A_H
// (A_H + B_H and A_H + D_B with a reaction term).  x holds the start vector.  Returns the
// iterations used, or -1 when the tolerance was not reached.  On return x is the M-normalised
// eigenvector with a positive sum, lam its Rayleigh quotient and g = |integral of x| (= G(x)).
__device__ __noinline__ int lobpcg(CoarseWS& ws, int n, double tol, int maxit, int nu, float omega, double* red, EigShared* sh,
                      double& lam, double& g) {
  const int ld = n + 1;
  const int nact = (n - 1) * n;  // threads for_interior gives work to
  const double hm = 1.0 / (12.0 * n * n);
  const double* __restrict__ wx = ws.wx;
  const double* __restrict__ wy = ws.wy;
  const double* __restrict__ rx = ws.rx;
  const double* __restrict__ ry = ws.ry;
  const double* __restrict__ rd = ws.rd;
  // the operator A (+ B): stiffness and, with a reaction term, the reaction's seven-point form
  auto opA = [&](const double* u, int p) {
    const double au = stiff<double, double>(wx, wy, u, p, ld);
    return rx ? au + hm * react7<double, double>(rx, ry, rd, u, p, ld) : au;
  };
  auto applyAM = [&](const double* u, double* Au, double* Mu, double& uAu, double& uMu) {
    double acc[2] = {0.0, 0.0}, o[2];
    for_interior(n, [&](int p, int, int) {
      const double au = opA(u, p);
      const double mu = hm * mass7(u, p, ld);
      Au[p] = au;
      Mu[p] = mu;
      acc[0] += u[p] * au;
      acc[1] += u[p] * mu;
    });
    block_sum<2, double>(
        acc, o, red, [&](const double* t) { sh->scale = (double)rsqrtf((float)t[1]); sh->theta = t[0] / t[1]; }, nact);
    uAu = o[0];
    uMu = o[1];
  };
  double xAx, xMx;
  applyAM(ws.x, ws.Ax, ws.Mx, xAx, xMx);
  {
    const double s = sh->scale;
    for_interior(n, [&](int p, int, int) {
      ws.x[p] *= s;
      ws.Ax[p] *= s;
      ws.Mx[p] *= s;
    });
    __syncthreads();
  }
  double theta = sh->theta;
  bool have_p = false;
  int it = 0, conv = 0;
  for (; it < maxit; ++it) {
    {
      double acc[2] = {0.0, 0.0}, o[2];
      for_interior(n, [&](int p, int, int) {
        const double rv = ws.Ax[p] - theta * ws.Mx[p];
        ws.r32[p] = (float)rv;
        acc[0] += rv * rv;
        acc[1] += ws.Mx[p] * ws.Mx[p];
      });
      block_sum<2, double>(
          acc, o, red, [&](const double* t) { sh->conv = t[0] <= tol * tol * theta * theta * t[1]; }, nact);
      if (sh->conv) {
        conv = 1;
        break;
      }
    }
    vcycle<float>(ws.mg, ws.r32, ws.w32, omega, nullptr, nu);
    for_interior(n, [&](int p, int, int) { ws.w[p] = (double)ws.w32[p]; });
    __syncthreads();
    double g[12];
    {
      double acc[12];
      for (int i = 0; i < 12; ++i) acc[i] = 0.0;
      for_interior(n, [&](int p, int, int) {
        const double aw = opA(ws.w, p);
        const double mw = hm * mass7(ws.w, p, ld);
        ws.Aw[p] = aw;
        ws.Mw[p] = mw;
        const double wv = ws.w[p], xv = ws.x[p];
        acc[0] += wv * aw;
        acc[1] += wv * mw;
        acc[2] += xv * aw;
        acc[3] += xv * mw;
        acc[4] += xv * ws.Ax[p];
        acc[5] += xv * ws.Mx[p];
        if (have_p) {
          const double pv = ws.p[p];
          acc[6] += pv * aw;
          acc[7] += pv * mw;
          acc[8] += xv * ws.Ap[p];
          acc[9] += xv * ws.Mp[p];
          acc[10] += pv * ws.Ap[p];
          acc[11] += pv * ws.Mp[p];
        }
      });
      const bool hp = have_p;
      block_sum<12, double>(acc, g, red, [&](const double* gg) {
        // Gram matrices of the basis [x, w, p]
        double GA[3][3], GM[3][3];
        GA[0][0] = gg[4];
        GM[0][0] = gg[5];
        GA[1][1] = gg[0];
        GM[1][1] = gg[1];
        GA[0][1] = GA[1][0] = gg[2];
        GM[0][1] = GM[1][0] = gg[3];
        GA[2][2] = gg[10];
        GM[2][2] = gg[11];
        GA[1][2] = GA[2][1] = gg[6];
        GM[1][2] = GM[2][1] = gg[7];
        GA[0][2] = GA[2][0] = gg[8];
        GM[0][2] = GM[2][0] = gg[9];
        const int kk = hp ? 3 : 2;
        const double th0 = GA[0][0] / GM[0][0];  // Rayleigh quotient of the current x
        float As[3][3], Mf[3][3];
        for (int i = 0; i < kk; ++i)
          for (int j = 0; j < kk; ++j) {
            As[i][j] = (float)(GA[i][j] - th0 * GM[i][j]);
            Mf[i][j] = (float)GM[i][j];
          }
        float cf[3], mu;
        const int k = rayleigh_ritz_shifted(As, Mf, kk, cf, mu);
        if (k > 0) {
          if (cf[0] < 0) {
            cf[0] = -cf[0];
            cf[1] = -cf[1];
            cf[2] = -cf[2];
          }
          // Rayleigh quotient of the new iterate from the FP64 Gram matrices; approximate
          // normalisations (the Gram matrices are recomputed every iteration)
          const double c0 = cf[0], c1 = cf[1], c2 = k > 2 ? cf[2] : 0.0;
          double ca = 0.0, cm = 0.0;
          const double cv[3] = {c0, c1, c2};
          for (int i = 0; i < k; ++i)
            for (int j = 0; j < k; ++j) {
              ca += cv[i] * GA[i][j] * cv[j];
              cm += cv[i] * GM[i][j] * cv[j];
            }
          const float xs = rsqrtf((float)cm);
          const float pp = cf[1] * cf[1] * Mf[1][1] + 2 * cf[1] * (k > 2 ? cf[2] : 0.0f) * Mf[1][2] +
                           (k > 2 ? cf[2] * cf[2] * Mf[2][2] : 0.0f);
          const float ps = pp > 0 ? rsqrtf(pp) : 0.0f;
          sh->pc[0] = cf[1] * ps;
          sh->pc[1] = (k > 2 ? cf[2] : 0.0f) * ps;
          sh->c[0] = c0 * xs;
          sh->c[1] = c1 * xs;
          sh->c[2] = c2 * xs;
          sh->theta = ca / cm;
        }
        sh->k = k;
      }, nact);
    }
    const int k = sh->k;
    if (k == 0) break;
    const double c0 = sh->c[0], c1 = sh->c[1], c2 = sh->c[2], q0 = sh->pc[0], q1 = sh->pc[1];
    const bool use_p = have_p && k > 2;
    for_interior(n, [&](int p, int, int) {
      const double xv = ws.x[p], axv = ws.Ax[p], mxv = ws.Mx[p];
      const double wv = ws.w[p], awv = ws.Aw[p], mwv = ws.Mw[p];
      const double pv = use_p ? ws.p[p] : 0.0, apv = use_p ? ws.Ap[p] : 0.0, mpv = use_p ? ws.Mp[p] : 0.0;
      ws.x[p] = c0 * xv + c1 * wv + c2 * pv;
      ws.Ax[p] = c0 * axv + c1 * awv + c2 * apv;
      ws.Mx[p] = c0 * mxv + c1 * mwv + c2 * mpv;
      ws.p[p] = q0 * wv + q1 * pv;
      ws.Ap[p] = q0 * awv + q1 * apv;
      ws.Mp[p] = q0 * mwv + q1 * mpv;
    });
    __syncthreads();
    theta = sh->theta;
    have_p = true;
  }
  // final: fresh operator application, normalisation, sign
  double xA, xM;
  applyAM(ws.x, ws.Ax, ws.Mx, xA, xM);
  double sacc[1] = {0.0}, so[1];
  for_interior(n, [&](int p, int, int) { sacc[0] += ws.x[p]; });
  block_sum<1, double>(sacc, so, red, [&](const double* t) {
    sh->scale = (t[0] < 0 ? -1.0 : 1.0) / sqrt(xM);
    sh->theta = xA / xM;
    // the integral of a P1 function with zero boundary values is h^2 times the sum of its nodal
    // values (each interior hat function integrates to h^2)
    sh->c[0] = fabs(t[0]) / ((double)n * n * sqrt(xM));
  }, nact);
  const double sc = sh->scale;
  for_interior(n, [&](int p, int, int) { ws.x[p] *= sc; });
  __syncthreads();
  lam = sh->theta;
  g = sh->c[0];
  return conv ? it : -1;
}

// Block sum of NV double-floats (fixed order: deterministic); thread 0 runs ep(totals) before the closing
// barrier.  red as in block_sum.
template <int NV, class Ep>
__device__ __forceinline__ void block_sum_df(df (&v)[NV], double* red, Ep ep) {
  static_assert(NV <= 12, "block_sum_df reduces at most 12 values");
  df* part = reinterpret_cast<df*>(red);
  df* tot = part + kRedWarps * 12;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int base = 0, c = NV;
  DfButterfly<NV, 16>::run(v, lane, base, c);
  if (c >= 1) part[wid * NV + base] = v[0];
  __syncthreads();
  if (wid == 0) {
    if (lane < NV) {
      df s = part[lane];
      for (int w = 1; w < nw; ++w) s = df_add(s, part[w * NV + lane]);
      tot[lane] = s;
    }
    __syncwarp();
    if (lane == 0) {
      df t[NV];
#pragma unroll
      for (int i = 0; i < NV; ++i) t[i] = tot[i];
      ep(t);
    }
  }
  __syncthreads();
}

// 12 / h^2 times the reaction's value at node p, 2 x sum r_q - sum r_q d_q over the six neighbours, from the
// edge weights r (pairs) and the differences d_q = x_p - x_q
__device__ __forceinline__ df reaction_df(const float* rx, const float* ry, const float* rd, const float* rxl,
                                          const float* ryl, const float* rdl, int p, int ld, df x, df dE, df dW, df dN,
                                          df dS, df dNE, df dSW) {
  const df w[6] = {{rx[p], rxl[p]},           {rx[p - 1], rxl[p - 1]}, {ry[p], ryl[p]},
                   {ry[p - ld], ryl[p - ld]}, {rd[p], rdl[p]},         {rd[p - ld - 1], rdl[p - ld - 1]}};
  const df d[6] = {dE, dW, dN, dS, dNE, dSW};
  df rs = {0.0f, 0.0f}, rdq = {0.0f, 0.0f};
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    df_acc(rs, w[k]);
    df_acc(rdq, df_mul(w[k], d[k]));
  }
  rs = fast_two_sum(rs.h, rs.l);
  df bx = df_mul(rs, df{2.0f * x.h, 2.0f * x.l});
  df_acc(bx, df_neg(rdq));
  return fast_two_sum(bx.h, bx.l);
}

struct Eig32Shared {
  df theta;        // shift of the residual: the predicted Rayleigh quotient
  float delta;     // x.r / x.Mx: the Rayleigh quotient is theta + delta
  float xmx;
  float al, be;    // x += al w + be p
  int conv, ok;
  double lam, g, scale;
};

// Rayleigh-Ritz on the basis [x, w, p] (k = 3; [x, w] for k = 2) for lobpcg32, by one thread: the smallest
// eigenpair of the pencil shifted by the Rayleigh quotient of x, so that x.Kx = 0.  With the scaled x as
// first unit vector the eigenvector is (1, y), y = -C(mu)^{-1} g(mu), where C and g are the other block and
// the coupling of K - mu M; the iteration mu <- Rayleigh quotient of (1, y) is Newton's on the Schur
// complement, which decreases and is concave left of C's eigenvalues, so from mu = 0 it converges
// monotonically to the smallest eigenvalue and quadratically (the shift is small by then).  Returns
// false when C(0) is not safely positive definite or w and p are nearly parallel.
__device__ bool ritz_newton(float m00, const float b[2], const float m0[2], const float K[3], const float M[3], int k,
                            float& al, float& be, float& mu) {
  // K, M: entries 11, 12, 22 of the block on w, p
  if (!(m00 > 0.0f) || !(M[0] > 0.0f) || (k > 2 && !(M[2] > 0.0f))) return false;
  const float d0 = rsqrtf(m00), d1 = rsqrtf(M[0]), d2 = k > 2 ? rsqrtf(M[2]) : 0.0f;
  const float m12 = k > 2 ? M[1] * d1 * d2 : 0.0f, k11 = K[0] * d1 * d1;
  const float k12 = k > 2 ? K[1] * d1 * d2 : 0.0f, k22 = k > 2 ? K[2] * d2 * d2 : 1.0f;
  const float m22 = k > 2 ? 1.0f : 0.0f;
  const float k01 = b[0] * d0 * d1, k02 = k > 2 ? b[1] * d0 * d2 : 0.0f;
  const float m01 = m0[0] * d0 * d1, m02 = k > 2 ? m0[1] * d0 * d2 : 0.0f;
  if (!(1.0f - m12 * m12 > 1e-5f)) return false;
  if (!(k11 > 0.0f) || !(k22 > 0.0f) || !(k11 * k22 - k12 * k12 > 1e-5f * k11 * k22)) return false;
  float y1 = 0.0f, y2 = 0.0f, m = 0.0f;
#pragma unroll 1
  for (int it = 0; it < 6; ++it) {
    const float c11 = k11 - m, c12 = k12 - m * m12, c22 = k22 - m * m22;
    const float g1 = k01 - m * m01, g2 = k02 - m * m02;
    const float idet = 1.0f / (c11 * c22 - c12 * c12);
    y1 = (c12 * g2 - c22 * g1) * idet;
    y2 = (c12 * g1 - c11 * g2) * idet;
    const float num = 2.0f * (k01 * y1 + k02 * y2) + k11 * y1 * y1 + 2.0f * k12 * y1 * y2 + (k > 2 ? k22 * y2 * y2 : 0.0f);
    const float den = 1.0f + 2.0f * (m01 * y1 + m02 * y2) + y1 * y1 + 2.0f * m12 * y1 * y2 + m22 * y2 * y2;
    if (!(den > 1e-3f)) return false;
    const float mn = num / den;
    const bool done = fabsf(mn - m) <= 1e-6f * fabsf(mn);
    m = mn;
    if (done) break;
  }
  mu = m;
  al = y1 * d1 / d0;
  be = y2 * d2 / d0;
  return isfinite(al) && isfinite(be) && isfinite(mu);
}

// LOBPCG of the FP32 kernel: as lobpcg, with only the iterate and its residual r = A x - theta M x in more
// than FP32.  The residual is formed afresh from x in double-floats each iteration (differences first, as
// in the streaming tier's residual), with theta the Rayleigh quotient predicted by the last
// Rayleigh-Ritz step; x.r gives the exact quotient.  Everything else -- the preconditioned residual w
// (an FP32 V-cycle), the last correction p, their images and the Gram matrix of the shifted pencil --
// only steers the correction x += al w + be p, whose FP32 rounding the next residual corrects.  The
// FP64 form keeps nine FP64 vectors (one sample of mesh 1/32 per SM) and executes about 60 FP64
// instructions per node and iteration, at sixteen clocks of an SM each; this one needs about 300 FP32
// instructions and half the memory.  8,192 direct eigensolves on mesh 1/32 (a window of
// the six-level workload's level 0): 15.8 -> 5.3 ms.  On return xh + xl is the M-normalised eigenvector with a positive sum, lam its Rayleigh quotient, g =
// |integral of x|; the result is the iterations used or -1.
__device__ __noinline__ int lobpcg32(CoarseWS32& ws, int n, double tol, int maxit, int nu, float omega, double* red,
                                     Eig32Shared* sh, double lam0, double& lam, double& g) {
  const int ld = n + 1;
  const double hm64 = 1.0 / (12.0 * n * n);
  const float h2 = 1.0f / ((float)n * (float)n), hm = h2 / 12.0f;
  const df hmd = {(float)hm64, (float)(hm64 - (double)(float)hm64)};
  const float* __restrict__ wxh = ws.mg.wx[0];
  const float* __restrict__ wyh = ws.mg.wy[0];
  float* __restrict__ aw = ws.mg.t[0];  // free outside the V-cycle
  if (threadIdx.x == 0) {
    sh->theta = df_split(lam0);
    sh->conv = 0;
  }
  __syncthreads();
  const float tol2 = (float)(tol * tol);
  // r = A x - theta M x; sums x.r, x.x, x.S6, r.r, r.Mx, Mx.Mx; last: the Rayleigh quotient in FP64
  auto residual = [&](bool last) {
    const df th = sh->theta;
    df c2 = df_mul(th, h2), c12 = df_mul(th, hmd);
    c12 = fast_two_sum(c12.h, c12.l);
    df acc[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) acc[k] = {0.0f, 0.0f};
    for_interior(n, [&](int p, int, int) {
      auto X = [&](int q) { return df{ws.xh[q], ws.xl[q]}; };
      const df x = X(p);
      const df dE = df_sub(x, X(p + 1)), dW = df_sub(x, X(p - 1)), dN = df_sub(x, X(p + ld)), dS = df_sub(x, X(p - ld));
      const df dNE = df_sub(x, X(p + ld + 1)), dSW = df_sub(x, X(p - ld - 1));
      df r = df_mul(df{wxh[p], ws.wxl[p]}, dE);
      df_acc(r, df_mul(df{wxh[p - 1], ws.wxl[p - 1]}, dW));
      df_acc(r, df_mul(df{wyh[p], ws.wyl[p]}, dN));
      df_acc(r, df_mul(df{wyh[p - ld], ws.wyl[p - ld]}, dS));
      df s6 = dE;
      df_acc(s6, dW);
      df_acc(s6, dN);
      df_acc(s6, dS);
      df_acc(s6, dNE);
      df_acc(s6, dSW);
      s6 = fast_two_sum(s6.h, s6.l);
      if (ws.rx)
        df_acc(r, df_mul(hmd, reaction_df(ws.rx, ws.ry, ws.rd, ws.rxl, ws.ryl, ws.rdl, p, ld, x, dE, dW, dN, dS, dNE, dSW)));
      df_acc(r, df_neg(df_mul(c2, x)));
      df_acc(r, df_mul(c12, s6));
      r = fast_two_sum(r.h, r.l);
      ws.r[p] = r.h;
      const float mx = h2 * (x.h - s6.h * (1.0f / 12.0f));
      df_acc(acc[0], df_mul(r, x));
      df_acc(acc[1], df_mul(x, x));
      df_acc(acc[2], df_mul(x, s6));
      acc[3].h = fmaf(r.h, r.h, acc[3].h);
      acc[4].h = fmaf(r.h, mx, acc[4].h);
      acc[5].h = fmaf(mx, mx, acc[5].h);
    });
    block_sum_df<6>(acc, red, [&](const df* t) {
      const float xmx = h2 * (t[1].h - t[2].h * (1.0f / 12.0f));
      const float d = (t[0].h + t[0].l) / xmx;
      sh->xmx = xmx;
      sh->delta = d;
      const float th1 = th.h + d, rr = t[3].h - 2.0f * d * t[4].h + d * d * t[5].h;
      sh->conv = rr <= tol2 * th1 * th1 * t[5].h;
      if (last || sh->conv) {
        const double m = (df_double(t[1]) - df_double(t[2]) / 12.0) / ((double)n * n);
        sh->lam = df_double(th) + df_double(t[0]) / m;
        sh->scale = 1.0 / sqrt(m);
      }
    });
  };
  // the shift of a start vector is only a guess: one pass measures it
  residual(false);
  if (threadIdx.x == 0) sh->theta = df_add(sh->theta, df{sh->delta, 0.0f});
  __syncthreads();
  bool have_p = false;
  int it = 0, conv = 0, evaluated = 0;
  for (;; ++it) {
    residual(it == maxit);
    if (sh->conv) conv = 1;
    if (conv || it == maxit) {
      evaluated = 1;
      break;
    }
    vcycle<float>(ws.mg, ws.r, ws.w, omega, nullptr, nu);
    {
      const float th = sh->theta.h + sh->delta;
      float acc[10];
      double o[10];
#pragma unroll
      for (int i = 0; i < 10; ++i) acc[i] = 0.0f;
      for_interior(n, [&](int p, int, int) {
        float a = stiff<float, float>(wxh, wyh, ws.w, p, ld);
        if (ws.rx) a += hm * react7<float, float>(ws.rx, ws.ry, ws.rd, ws.w, p, ld);
        const float m = hm * mass7(ws.w, p, ld);
        aw[p] = a;
        ws.mw[p] = m;
        const float wv = ws.w[p], xv = ws.xh[p], rv = ws.r[p], kw = a - th * m;
        acc[0] += wv * rv;
        acc[1] += xv * m;
        acc[2] += wv * kw;
        acc[3] += wv * m;
        if (have_p) {
          const float pv = ws.p[p], pm = ws.mp[p];
          acc[4] += pv * rv;
          acc[5] += xv * pm;
          acc[6] += pv * kw;
          acc[7] += pv * m;
          acc[8] += pv * (ws.ap[p] - th * pm);
          acc[9] += pv * pm;
        }
      });
      const bool hp = have_p;
      block_sum<10, float>(acc, o, red, [&](const double* t) {
        float v[10];
        for (int i = 0; i < 10; ++i) v[i] = (float)t[i];
        const float dl = sh->delta;
        const float b[2] = {v[0] - dl * v[1], v[4] - dl * v[5]}, m0[2] = {v[1], v[5]};
        const float K[3] = {v[2], v[6], v[8]}, M[3] = {v[3], v[7], v[9]};
        float al = 0.0f, be = 0.0f, mu = 0.0f;
        bool ok = (hp && ritz_newton(sh->xmx, b, m0, K, M, 3, al, be, mu)) || ritz_newton(sh->xmx, b, m0, K, M, 2, al, be, mu);
        if (!ok) {
          const float GA[3][3] = {{0.0f, b[0], b[1]}, {b[0], K[0], K[1]}, {b[1], K[1], K[2]}};
          const float GM[3][3] = {{sh->xmx, m0[0], m0[1]}, {m0[0], M[0], M[1]}, {m0[1], M[1], M[2]}};
          float c[3];
          const int k = rayleigh_ritz_shifted(GA, GM, hp ? 3 : 2, c, mu);
          ok = k > 0 && c[0] != 0.0f;
          if (ok) {
            al = c[1] / c[0];
            be = k > 2 ? c[2] / c[0] : 0.0f;
          }
        }
        sh->al = al;
        sh->be = be;
        sh->ok = ok;
        if (ok) sh->theta = df_add(sh->theta, two_sum(dl, mu));
      });
    }
    if (!sh->ok) break;
    const float al = sh->al, be = sh->be;
    const bool use_p = have_p && be != 0.0f;
    for_interior(n, [&](int p, int, int) {
      const float pv = use_p ? ws.p[p] : 0.0f, apv = use_p ? ws.ap[p] : 0.0f, mpv = use_p ? ws.mp[p] : 0.0f;
      const float d = fmaf(al, ws.w[p], be * pv);
      const df x = df_add(df{ws.xh[p], ws.xl[p]}, df{d, 0.0f});
      ws.xh[p] = x.h;
      ws.xl[p] = x.l;
      ws.p[p] = d;
      ws.ap[p] = fmaf(al, aw[p], be * apv);
      ws.mp[p] = fmaf(al, ws.mw[p], be * mpv);
    });
    __syncthreads();
    have_p = true;
  }
  if (!evaluated) residual(true);
  // normalisation and sign; the integral of a P1 function with zero boundary values is h^2 times the
  // sum of its nodal values
  df sacc[1] = {{0.0f, 0.0f}};
  for_interior(n, [&](int p, int, int) { df_acc(sacc[0], df{ws.xh[p], ws.xl[p]}); });
  block_sum_df<1>(sacc, red, [&](const df* t) {
    const double sum = df_double(t[0]);
    sh->g = fabs(sum) * sh->scale / ((double)n * n);
    if (sum < 0.0) sh->scale = -sh->scale;
  });
  const df sc = df_split(sh->scale);
  for_interior(n, [&](int p, int, int) {
    const df v = df_mul(df{ws.xh[p], ws.xl[p]}, sc), x = fast_two_sum(v.h, v.l);
    ws.xh[p] = x.h;
    ws.xl[p] = x.l;
  });
  __syncthreads();
  lam = sh->lam;
  g = sh->g;
  return conv ? it : -1;
}

// MINRES iterations per correction of a solve on the coarse mesh itself.  Ten to thirteen reduce a residual by the 1e-4 asked for;
// where the shift nearly meets the eigenvalue they leave what r has along the near-null direction, and iterations
// beyond run into FP32's idea of that eigenvalue: the correction grows without bound (450 ||u_H||, residual 1e2
// to 1e4 ||b||).  With 24 one sample in 150 needed the FP64 solve behind it, and calls of few samples waited
// for it: 128 solves on mesh 1/64 7.2 ms, on 1/128 31.7 ms.  With 12 none of 5,000 did: 2.5 and 12.7 ms (FP64 throughout: 4.6 and
// 20.0); 8,192 samples of the first test problem's level 1 7.85 -> 6.83 ms; with 10, 14, 16 and 18: 6.81, 6.94, 7.32, 7.78.
constexpr int kNearInner = 12;

// The coarse eigenvector as the fine solves read it: FP64 values, or double-float pairs.
struct CoarseVec {
  const double* d;
  const float *h, *l;
  __device__ double operator[](int q) const { return d ? d[q] : (double)h[q] + (double)l[q]; }
  __device__ df pair(int q) const { return d ? df_split(d[q]) : df{h[q], l[q]}; }
};

// The operator of a sample in FP32 with the low parts of its finest weights, coefficients times 2^-k: hierarchy and
// reaction weights of a coarse (CoarseWS32) or fine (FineWS<float>) workspace
template <typename WS>
__device__ __forceinline__ void operator32(WS& ws, int n, const double* a, const double* rb, int k) {
  build_mg<float>(ws.mg, a, n, rb, ws.wxl, ws.wyl, k);
  if (rb) reaction_weights<float, double>(n, rb, rb + (size_t)n * n, ws.rx, ws.ry, ws.rd, ws.rxl, ws.ryl, ws.rdl, k);
}
// the same out of line: inlined into twogrid_fine it costs registers that the iterations then spill (first test
// problem's level 1, 8,192 samples: 7.96 ms inline, 7.84 out of line)
template <typename WS>
__device__ __noinline__ void operator32_scaled(WS& ws, int n, const double* a, const double* rb, int k) {
  operator32(ws, n, a, rb, k);
}

// the operator of the FP64 eigensolver: FP32 hierarchy, FP64 weights
__device__ __forceinline__ void operator64(CoarseWS& ws, int n, const double* a, const double* rb, int k) {
  build_mg<float>(ws.mg, a, n, rb, nullptr, nullptr, k);
  weights_from_cells<double, double>(n, a, a + (size_t)n * n, ws.wx, ws.wy, nullptr, nullptr, k);
  if (rb) reaction_weights<double, double>(n, rb, rb + (size_t)n * n, ws.rx, ws.ry, ws.rd, nullptr, nullptr, nullptr, k);
}
__device__ __noinline__ void operator64_scaled(CoarseWS& ws, int n, const double* a, const double* rb, int k) {
  operator64(ws, n, a, rb, k);
}

// MINRES scalars, owned by thread 0 and read by all threads after each reduction.  The
// recurrences run in the inner precision T (FP32 on the mixed path); the refinement's scalars are FP64.
template <typename T>
struct MinresShared {
  T gam, gam_old, eta, eta0, c, c_old, s, s_old;
  T ig;           // 1 / gamma_j
  T c1, c2;       // v_new = q - c1 v - c2 v_old
  T cx, ia1, a2, a3;  // pending w / x update
  T delta;
  T rs;           // 1 / ||r|| of the refinement residual
  double rnorm, bnorm;
  double knorm, xnorm;  // ||A - sigma M|| bound and ||x|| for the residual's rounding floor
  double xax, xmx;      // x.Ax and x.Mx of the last residual pass (the Rayleigh quotient)
  double xsum;          // sum of the nodal values of x in that pass (h^2 xsum = integral of x)
  double scale;         // 2^ks: the solve is the problem times 2^-ks
  double tau;           // factor of the right-hand side (1 except in a solve on the coarse mesh itself)
  int done, breakdown;
};

// Residual target of the refinement: tol relative to ||b||, but never below a small multiple of
// the rounding floor eps (||K|| ||x|| + ||b||) of an FP64 residual (double-floats stop short of it by the lack of
// progress; on fine meshes the
// near-singular shifted system puts that floor above 1e-7 ||b||).
__host__ __device__ inline double residual_target(double tol, double bnorm, double knorm, double xnorm, double f) {
  const double floor_ = f * 2.220446049250313e-16 * (knorm * xnorm + bnorm);
  const double t = tol * bnorm;
  return t > floor_ ? t : floor_;
}

// ---------------------------------------------------------------------------------------------
// two-grid update on the fine mesh n: returns the Rayleigh quotient of the solution of
// (A - sigma M) w = M P u_H (A + B - sigma M with the reaction coefficient rb), and in gq the
// functional G(w) = |integral of w| / ||w||_L2.  iters / outer report the inner MINRES iterations
// and refinement steps; flags receives kFlag* bits.
template <typename T>
__device__ __noinline__ double twogrid_fine(FineWS<T>& ws, char* fine_base, int n, const double* __restrict__ a,
                               const double* __restrict__ rb, const CoarseVec uH, int nc, double sigma,
                               const SampleLaunch& P, double* red, MinresShared<T>* ms, int& iters, int& outer,
                               int& flags, double& gq) {
  constexpr bool kF32 = sizeof(T) == sizeof(float);
  // A solve on the coarse mesh itself (a longer truncation on the mesh of the coarse pair): see `near` below
  const bool near = kF32 && n == nc;
  const int ld = n + 1;
  __syncthreads();
  if (threadIdx.x == 0) {
    Carver f(fine_base);
    carve_fine<T>(f, n, ws, rb != nullptr);
  }
  __syncthreads();
  const double hm = 1.0 / (12.0 * n * n);
  if constexpr (kF32) {
    float* const pr[4] = {ws.xh, ws.xl, ws.bh, ws.bl};
    for (float* v : pr) zero_vec(v, n);
  } else {
    zero_vec(ws.x64, n);
    zero_vec(ws.b64, n);
  }
  zero_vec(ws.vo, n);
  zero_vec(ws.v, n);
  zero_vec(ws.z, n);
  zero_vec(ws.zn, n);
  if (rb) {
    zero_vec(ws.rx, n);
    zero_vec(ws.ry, n);
    zero_vec(ws.rd, n);
  }
  zero_mg(ws.mg);
  // FP32 kernel: everything below is the problem times 2^-ks (see mq_device.cuh)
  const int ks = kF32 ? scale_of_shift(sigma) : 0;
  sigma *= pow2(-ks);
  __syncthreads();
  CellCheck cells;
  cells.look(n, a, rb);
  if constexpr (kF32) {
    operator32_scaled(ws, n, a, rb, ks);
  } else {
    build_mg<T>(ws.mg, a, n, rb);
    if (rb) reaction_weights<T, double>(n, rb, rb + (size_t)n * n, ws.rx, ws.ry, ws.rd);
  }
  if (!cells.finish(red)) flags |= kFlagBadCoef;
  if (threadIdx.x == 0) {
    // ||A + B - sigma M||_inf <= 8 max a + (max b + sigma) h^2 (row sums of the edge form, of the
    // reaction and of the mass)
    ms->knorm = 8.0 * (pow2(-ks) * cell_bound(cells.amax)) + (pow2(-ks) * cell_bound(cells.bmax) + sigma) / ((double)n * n);
    ms->scale = pow2(ks);
    ms->xnorm = 0.0;
    ms->xax = ms->xmx = 0.0;
    ms->tau = 1.0;
  }
  __syncthreads();
  // FP64 kernel: the operator of the residual from the FP64 weights of level 0
  const double* wx64 = (const double*)ws.mg.wx[0];
  const double* wy64 = (const double*)ws.mg.wy[0];
  auto K64 = [&](const double* x, int p) {
    double k = stiff<double, double>(wx64, wy64, x, p, ld);
    if (rb) k += hm * react7<double, double>((const double*)ws.rx, (const double*)ws.ry, (const double*)ws.rd, x, p, ld);
    return k;
  };
  const df hmd = {(float)hm, (float)(hm - (double)(float)hm)};
  // FP32 kernel: the residual of the current x in double-floats (as the streaming tier's: see k_residual4), and
  // with it x.Kx, x.x, x.S6 and sum x.  With `near` the right-hand side is tau b with tau = x.Kx / x.b,
  // r orthogonal to x: a solve on the coarse mesh itself has its shift at an eigenvalue
  // of a nearby operator, K w = b a solution w that is almost a multiple of u_H and may be
  // arbitrarily long, and only its direction matters.  Written as w = (u_H + v) / tau the unknown
  // v is as small as the change of the coefficient, and FP32 corrections converge for any distance
  // of the shift from the eigenvalue (x soon is the near-null direction itself, and r orthogonal
  // to it leaves that direction out of the correction).  The residual of w relative to ||b|| is ||tau b - K (u_H + v)|| / (|tau| ||b||).
  auto residual32 = [&](bool first_pass) {
    if constexpr (kF32) {
      const double c12d = sigma / ((double)n * n);
      const df c12 = df_split(c12d), cs = df_split(sigma * hm);
      df acc[6];
#pragma unroll
      for (int k = 0; k < 6; ++k) acc[k] = {0.0f, 0.0f};
      const float* __restrict__ wxh = (const float*)ws.mg.wx[0];
      const float* __restrict__ wyh = (const float*)ws.mg.wy[0];
      for_interior(n, [&](int p, int, int) {
        auto X = [&](int q) { return df{ws.xh[q], ws.xl[q]}; };
        const df x = X(p);
        const df dE = df_sub(x, X(p + 1)), dW = df_sub(x, X(p - 1)), dN = df_sub(x, X(p + ld)), dS = df_sub(x, X(p - ld));
        const df dNE = df_sub(x, X(p + ld + 1)), dSW = df_sub(x, X(p - ld - 1));
        df k = df_mul(df{wxh[p], ws.wxl[p]}, dE);
        df_acc(k, df_mul(df{wxh[p - 1], ws.wxl[p - 1]}, dW));
        df_acc(k, df_mul(df{wyh[p], ws.wyl[p]}, dN));
        df_acc(k, df_mul(df{wyh[p - ld], ws.wyl[p - ld]}, dS));
        df s6 = dE;
        df_acc(s6, dW);
        df_acc(s6, dN);
        df_acc(s6, dS);
        df_acc(s6, dNE);
        df_acc(s6, dSW);
        s6 = fast_two_sum(s6.h, s6.l);
        if (ws.rx) df_acc(k, df_mul(hmd, reaction_df(ws.rx, ws.ry, ws.rd, ws.rxl, ws.ryl, ws.rdl, p, ld, x, dE, dW, dN, dS, dNE, dSW)));
        df_acc(k, df_neg(df_mul(c12, x)));
        df_acc(k, df_mul(cs, s6));
        k = fast_two_sum(k.h, k.l);
        const df bv = {ws.bh[p], ws.bl[p]};
        if (near) {
          ws.zn[p] = k.h;
          ws.vo[p] = k.l;
          df_acc(acc[5], df_mul(bv, x));
        } else {
          df r = bv;
          df_acc(r, df_neg(k));
          const float rf = r.h + r.l;
          ws.v[p] = rf;
          acc[0].h = fmaf(rf, rf, acc[0].h);
        }
        df_acc(acc[1], df_mul(x, x));
        df_acc(acc[2], df_mul(x, k));
        df_acc(acc[3], df_mul(x, s6));
        df_acc(acc[4], x);
      });
      auto finish = [&](double rr) {
        const double rnew = sqrt(rr);
        // no progress: stop refining (not after the first step, whose FP32 rounding noise can
        // leave a residual above ||b|| on fine meshes)
        ms->done = !first_pass && outer > 0 && !(rnew < 0.5 * ms->rnorm);
        ms->rnorm = rnew;
        ms->rs = T(1.0 / rnew);
      };
      block_sum_df<6>(acc, red, [&](const df* t) {
        const double x2 = df_double(t[1]), xk = df_double(t[2]), x6 = df_double(t[3]);
        ms->xnorm = sqrt(x2);
        ms->xmx = (x2 - x6 / 12.0) / ((double)n * n);
        ms->xax = xk + sigma * ms->xmx;
        ms->xsum = df_double(t[4]);
        if (near)
          ms->tau = xk / df_double(t[5]);
        else
          finish(df_double(t[0]));
      });
      if (near) {
        const df tau = df_split(ms->tau);
        df acc1[1] = {{0.0f, 0.0f}};
        for_interior(n, [&](int p, int, int) {
          df r = df_mul(tau, df{ws.bh[p], ws.bl[p]});
          df_acc(r, df{-ws.zn[p], -ws.vo[p]});
          const float rf = r.h + r.l;
          ws.v[p] = rf;
          acc1[0].h = fmaf(rf, rf, acc1[0].h);
        });
        block_sum_df<1>(acc1, red, [&](const df* t) { finish(df_double(t[0])); });
      }
    }
  };
  // b = M P u_H  (P: P1 interpolation from the nested coarse mesh); x holds P u_H for a moment (with `near`
  // it stays there)
  {
    const int lr = ilog2(n / nc);
    const int rm = (1 << lr) - 1;
    const int ldc = nc + 1;
    const double inv = 1.0 / (double)(1 << lr);
    for_interior(n, [&](int p, int i, int j) {
      const int I = i >> lr, J = j >> lr;
      const int c0 = J * ldc + I;
      if constexpr (kF32) {
        const int ki = i & rm, kj = j & rm;
        const bool lower = ki >= kj;
        const df u00 = uH.pair(c0), u11 = uH.pair(c0 + ldc + 1), uc = uH.pair(lower ? c0 + 1 : c0 + ldc);
        const float s1 = (float)(lower ? ki : kj) * (float)inv, s2 = (float)(lower ? kj : ki) * (float)inv;
        const df v = df_add(df_add(u00, df_mul(df_sub(uc, u00), s1)), df_mul(df_sub(u11, uc), s2));
        ws.xh[p] = v.h;
        ws.xl[p] = v.l;
      } else {
        const double xi_ = (double)(i & rm) * inv, et = (double)(j & rm) * inv;
        double v;
        if (xi_ >= et)
          v = (1.0 - xi_) * uH[c0] + (xi_ - et) * uH[c0 + 1] + et * uH[c0 + ldc + 1];
        else
          v = (1.0 - et) * uH[c0] + (et - xi_) * uH[c0 + ldc] + xi_ * uH[c0 + ldc + 1];
        ws.x64[p] = v;
      }
    });
    __syncthreads();
    double acc[1] = {0.0}, o[1];
    float acc32[1] = {0.0f};
    for_interior(n, [&](int p, int, int) {
      if constexpr (kF32) {
        df m = df_mul(df{ws.xh[p], ws.xl[p]}, 6.0f);
        const int q[6] = {p + 1, p - 1, p + ld, p - ld, p + ld + 1, p - ld - 1};
#pragma unroll
        for (int k = 0; k < 6; ++k) df_acc(m, df{ws.xh[q[k]], ws.xl[q[k]]});
        df bv = df_mul(m, hmd);
        bv = fast_two_sum(bv.h, bv.l);
        ws.bh[p] = bv.h;
        ws.bl[p] = bv.l;
        ws.v[p] = bv.h;
        acc32[0] = fmaf(bv.h, bv.h, acc32[0]);
      } else {
        const double bv = hm * mass7(ws.x64, p, ld);
        ws.b64[p] = bv;
        ws.v[p] = T(bv);
        acc[0] += bv * bv;
      }
    });
    auto start = [&](const double* t) {
      ms->bnorm = ms->rnorm = sqrt(t[0]);
      ms->rs = T(1.0 / ms->rnorm);
    };
    if constexpr (kF32)
      block_sum<1, float>(acc32, o, red, start);
    else
      block_sum<1, double>(acc, o, red, start);
    if (!near) {
      for_interior(n, [&](int p, int, int) {
        if constexpr (kF32)
          ws.xh[p] = ws.xl[p] = 0.0f;
        else
          ws.x64[p] = 0.0;
      });
      __syncthreads();
    } else {
      residual32(true);
    }
  }
  outer = 0;
  iters = 0;
  // with the shift within FP32 rounding of the eigenvalue, a correction cannot reduce what r has along the
  // near-null direction before x has turned into it: such solves end early and the next one goes on
  const bool early = near && P.max_inner_it > kNearInner;
  const int max_inner = early ? kNearInner : P.max_inner_it;
  const T sigm = T(sigma * hm);
  const T hmt = T(hm);
  const T om = T(P.omega);
  const T* twx = ws.mg.wx[0];
  const T* twy = ws.mg.wy[0];
  const T* trx = ws.rx;
  const T* try_ = ws.ry;
  const T* trd = ws.rd;
  for (; outer < P.max_outer; ++outer) {
    if (!(ms->rnorm > residual_target(P.tol_lin, fabs(ms->tau) * ms->bnorm, ms->knorm, ms->xnorm, 16.0))) break;
    // inner: MINRES on (A - sigma M) xi = r / ||r|| in precision T, preconditioned by the V-cycle;
    // v holds r (unscaled)
    const T rs = ms->rs;
    for_interior(n, [&](int p, int, int) {
      ws.v[p] *= rs;
      ws.vo[p] = T(0);
      ws.w[p] = T(0);
      ws.wo[p] = T(0);
    });
    __syncthreads();
    T* vo = ws.vo;
    T* v = ws.v;
    T* z = ws.z;
    T* zn = ws.zn;
    T* wo = ws.wo;
    T* w = ws.w;
    {
      T acc1[1] = {vcycle<T>(ws.mg, v, z, om, v, P.nu)};  // z = B^{-1} v and <v, z>
      double o1[1];
      block_sum<1, T>(acc1, o1, red, [&](const double* t) {
        const T t0 = T(t[0]);
        ms->breakdown = !(t0 > T(0));
        const T g = ms->breakdown ? T(1) : sqrt(t0);
        ms->gam = g;
        ms->eta = ms->eta0 = g;
        ms->gam_old = T(1);
        ms->c = ms->c_old = T(1);
        ms->s = ms->s_old = T(0);
        ms->ig = T(1) / g;
        ms->done = ms->breakdown;
      });
    }
    if (ms->breakdown) {
      flags |= kFlagBreakdown;
      break;
    }
    // x += ||r|| eta_j w_j as the directions come: no array for the sum over a solve
    const double rn = ms->rnorm;
    auto add_x = [&](int p, T cx, T wnew) {
      if constexpr (kF32) {
        const df x = df_add(df{ws.xh[p], ws.xl[p]}, df{cx * wnew, 0.0f});
        ws.xh[p] = x.h;
        ws.xl[p] = x.l;
      } else {
        ws.x64[p] += cx * wnew;
      }
    };
    int j = 0;
    bool pending = false;
    for (; j < max_inner && !ms->done; ++j) {
      // [pending w/x update of the previous iteration] + q = K z / gamma, delta; q takes the place of the
      // normalised z of the previous step, which only the update at the same node still reads
      {
        T acc1[1] = {T(0)};
        double o1[1];
        const T ig = ms->ig;
        const T ta1 = ms->ia1, ta2 = ms->a2, ta3 = ms->a3, tcx = T(rn * (double)ms->cx);
        const bool pend = pending;
        for_interior(n, [&](int p, int, int) {
          if (pend) {
            const T wnew = (zn[p] - ta3 * wo[p] - ta2 * w[p]) * ta1;
            wo[p] = wnew;
            add_x(p, tcx, wnew);
          }
          T kz = stiff<T, T>(twx, twy, z, p, ld) - sigm * mass7(z, p, ld);
          if (trx) kz += hmt * react7<T, T>(trx, try_, trd, z, p, ld);
          kz *= ig;
          zn[p] = kz;
          acc1[0] += kz * z[p];
        });
        block_sum<1, T>(acc1, o1, red, [&](const double* t) {
          const T delta = T(t[0]) * ms->ig;
          ms->c1 = delta * ms->ig;
          ms->c2 = ms->gam / ms->gam_old;
          ms->delta = delta;
        });
        if (pend) {
          T* tt = wo;
          wo = w;
          w = tt;
        }
      }
      // v_new = q - (delta/gam) v - (gam/gam_old) v_old ; z normalised in place
      {
        const T c1 = ms->c1, c2 = ms->c2, ig = ms->ig;
        for_interior(n, [&](int p, int, int) {
          vo[p] = zn[p] - c1 * v[p] - c2 * vo[p];
          z[p] *= ig;
        });
        __syncthreads();
        T* tt = vo;
        vo = v;
        v = tt;
      }
      {
        T acc1[1] = {vcycle<T>(ws.mg, v, zn, om, v, P.nu)};  // zn = B^{-1} v_new and <v_new, zn>
        double o1[1];
        const T tol = T(P.tol_inner);
        block_sum<1, T>(acc1, o1, red, [&](const double* t) {
          T gnew = T(t[0]);
          if (!(gnew >= T(0))) {
            ms->breakdown = 1;
            gnew = T(0);
          }
          gnew = sqrt(gnew);
          const T delta = ms->delta, gam = ms->gam;
          const T al0 = ms->c * delta - ms->c_old * ms->s * gam;
          const T al1 = sqrt(al0 * al0 + gnew * gnew);
          const T al2 = ms->s * delta + ms->c_old * ms->c * gam;
          const T al3 = ms->s_old * gam;
          const T ia1 = T(1) / al1;
          const T cn = al0 * ia1, sn = gnew * ia1;
          ms->cx = cn * ms->eta;
          ms->ia1 = ia1;
          ms->a2 = al2;
          ms->a3 = al3;
          ms->eta = -sn * ms->eta;
          ms->s_old = ms->s;
          ms->s = sn;
          ms->c_old = ms->c;
          ms->c = cn;
          ms->gam_old = gam;
          ms->gam = gnew;
          ms->ig = gnew > T(0) ? T(1) / gnew : T(0);
          ms->done = fabs(ms->eta) <= tol * ms->eta0 || gnew == T(0) || ms->breakdown;
        });
        T* tt = z;
        z = zn;
        zn = tt;  // z = z_{j+1} (unnormalised), zn = z_j (normalised)
        pending = true;
      }
    }
    if (pending) {
      const T ta1 = ms->ia1, ta2 = ms->a2, ta3 = ms->a3, tcx = T(rn * (double)ms->cx);
      for_interior(n, [&](int p, int, int) { add_x(p, tcx, (zn[p] - ta3 * wo[p] - ta2 * w[p]) * ta1); });
      __syncthreads();
    }
    iters += j;
    if (ms->breakdown) flags |= kFlagBreakdown;
    if (!ms->done && !early) flags |= kFlagLinNoConv;
    // r = b - (A - sigma M) x beyond FP32, stored (unscaled) in v.  The same pass forms x.Ax, x.Mx and sum(x): the
    // last one gives the Rayleigh quotient and the functional of the result
    if constexpr (kF32) {
      residual32(false);
    } else {
      double acc2[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, o2[5];
      for_interior(n, [&](int p, int, int) {
        const double xv = ws.x64[p];
        const double ax = K64(ws.x64, p);
        const double mx = hm * mass7(ws.x64, p, ld);
        const double rv = ws.b64[p] - (ax - sigma * mx);
        ws.v[p] = T(rv);
        acc2[0] += rv * rv;
        acc2[1] += xv * xv;
        acc2[2] += xv * ax;
        acc2[3] += xv * mx;
        acc2[4] += xv;
      });
      const int first = outer == 0;
      block_sum<5, double>(acc2, o2, red, [&](const double* t) {
        const double rnew = sqrt(t[0]);
        ms->xnorm = sqrt(t[1]);
        ms->xax = t[2];
        ms->xmx = t[3];
        ms->xsum = t[4];
        // no progress: stop refining (not after the first step, whose FP32 rounding noise can
        // leave a residual above ||b|| on fine meshes)
        ms->done = !first && !(rnew < 0.5 * ms->rnorm);
        ms->rnorm = rnew;
        ms->rs = T(1.0 / rnew);
      });
    }
    const int stalled = ms->done;
    if (stalled) {
      ++outer;
      break;
    }
  }
  // flagged only well above the target (or the rounding floor): the refinement may stop a little short
  if (!(ms->rnorm <= residual_target(fmax(1e-5, 10.0 * P.tol_lin), fabs(ms->tau) * ms->bnorm, ms->knorm, ms->xnorm, 256.0)))
    flags |= kFlagLinNoConv;
  // Rayleigh quotient and functional from the sums of the residual pass over the final iterate (FP64, or 48 bits)
  gq = fabs(ms->xsum) / ((double)n * n * sqrt(ms->xmx));
  return ms->scale * (ms->xax / ms->xmx);
}

// MAXT: threads per block at most.  Up to 256 threads the FP32 kernel is compiled for three blocks of 256 per SM (80
// registers): its phases are short and end in block-wide barriers, which other blocks then fill.
template <typename T, int MAXT>
__global__ void __launch_bounds__(MAXT, sizeof(T) == sizeof(float) && MAXT == 256 ? 3 : 1) sample_kernel(SampleLaunch P) {
  extern __shared__ __align__(16) char smem_dyn[];
  __shared__ double red[kRedSlots];
  __shared__ EigShared esh;
  __shared__ Eig32Shared esh32;
  __shared__ MinresShared<T> msh;
  // one of the two coarse workspaces is in use (e32 below)
  __shared__ union CoarseBoth {
    CoarseWS f64;
    CoarseWS32 f32;
    __device__ CoarseBoth() {}
  } both;
  CoarseWS& cws = both.f64;
  CoarseWS32& cws32 = both.f32;
  __shared__ FineWS<T> fws;
  char* base = P.use_smem ? smem_dyn : P.gscratch + (size_t)blockIdx.x * P.slab_bytes;
  size_t persist_bytes;
  const bool rxn = P.reaction != 0;
  const bool e32 = sizeof(T) == sizeof(float) && P.eig32;
  if (e32) {
    Carver c(base);
    CoarseWS32 tmp;
    carve_coarse32(c, P.nc, tmp, &persist_bytes, rxn);
    if (threadIdx.x == 0) cws32 = tmp;
  } else {
    Carver c(base);
    CoarseWS tmp;
    carve_coarse(c, P.nc, tmp, &persist_bytes, rxn);
    if (threadIdx.x == 0) cws = tmp;
  }
  char* fine_base = base + ((persist_bytes + 15) & ~(size_t)15);  // the fine workspace overlays the coarse one
  __syncthreads();
  const int nc = P.nc;
  const int cpr = (P.npts + P.chunk - 1) / P.chunk;
  const int nchunks = cpr * P.R;
  const size_t ncT = (size_t)2 * nc * nc, nfT = (size_t)2 * P.nf * P.nf, npT = (size_t)2 * P.np * P.np;
  // the persistent coarse eigenvector: zero once (its ring stays zero)
  if (e32) {
    zero_vec(cws32.xh, nc);
    zero_vec(cws32.xl, nc);
  } else {
    zero_vec(cws.uprev, nc);
  }
  __syncthreads();
  const CoarseVec uH = e32 ? CoarseVec{nullptr, cws32.xh, cws32.xl} : CoarseVec{cws.uprev, nullptr, nullptr};
  double lam_prev = 0.0;  // coarse eigenvalue of the previous point of the chain (not finite: nothing to start from)
  // a fine solve; one on the coarse mesh itself that FP32 corrections could not finish (the shift meets the
  // eigenvalue by accident) runs again in FP64, its workspace in global memory
  auto fine = [&](int n, const double* a, const double* rb, double lamH, int& it, int& outer, int& flags, double& gq) {
    int fl = 0;
    double v = 0.0;
    const bool f64 = sizeof(T) == sizeof(float) && n == P.nc && P.nc > kNear32Max;  // beyond the FP32 form's reach
    if (!f64) v = twogrid_fine<T>(fws, fine_base, n, a, rb, uH, P.nc, lamH, P, red, &msh, it, outer, fl, gq);
    if constexpr (sizeof(T) == sizeof(float)) {
      if (f64 || (n == P.nc && (fl & (kFlagLinNoConv | kFlagBreakdown)))) {
        Carver c(P.fscratch + (size_t)blockIdx.x * P.fslab_bytes);
        FineWS<double>& ws = *c.take<FineWS<double>>(1);
        MinresShared<double>* ms = c.take<MinresShared<double>>(1);
        char* base64 = (char*)c.take<double2>(1);
        fl &= kFlagBadCoef;
        v = twogrid_fine<double>(ws, base64, n, a, rb, uH, P.nc, lamH, P, red, ms, it, outer, fl, gq);
      }
    }
    flags |= fl;
    return v;
  };
  const float omega = (float)P.omega;
  for (int ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
    const int r = ch / cpr;
    const int k0 = (ch % cpr) * P.chunk;
    const int k1 = min(k0 + P.chunk, P.npts);
    for (int kk = k0; kk < k1; ++kk) {
      const size_t b = (size_t)r * P.npts + kk;
      int flags = 0;
      // ---- coarse eigenpair (Algorithm 1 step 1; Algorithm 2 steps 6-7), or, in the reuse scheme
      // across levels, the level-0 eigenpair of this point given in u_in / out[b][0]
      CoarseWS& cw = cws;
      double lamH, gH = 0.0;
      int eit = 0;
      const bool cold = kk == k0 || !isfinite(lam_prev);
      if (P.u_in) {
        const size_t Vc = gsz(nc);
        for_all(Vc, [&](size_t q) {
          const double v = P.u_in[b * Vc + q];
          if (e32) {
            const df d = df_split(v);
            cws32.xh[q] = d.h;
            cws32.xl[q] = d.l;
          } else {
            cw.uprev[q] = v;
          }
        });
        lamH = P.out[b * 4 + 0];
        __syncthreads();
        if (P.qoi && (P.direct_f || (P.np > 0 && P.direct_p && !P.prev_given))) {
          // G(u_H) of the given (M-normalised) eigenvector: h^2 |sum u| / sqrt(u^T M u)
          const double hmc = 1.0 / (12.0 * nc * nc);
          double acc[2] = {0.0, 0.0}, o[2];
          for_interior(nc, [&](int p, int, int) {
            const int ldc = nc + 1;
            acc[0] += uH[p];
            acc[1] += uH[p] * hmc * (6.0 * uH[p] + (uH[p + 1] + uH[p - 1]) + (uH[p + ldc] + uH[p - ldc]) +
                                     (uH[p + ldc + 1] + uH[p - ldc - 1]));
          });
          block_sum<2, double>(acc, o, red);
          gH = fabs(o[0]) / ((double)nc * nc * sqrt(o[1]));
        }
      } else if (e32) {
        // the fine solves of the previous point reused this memory: clear the coarse vectors (the rings
        // must be zero; interiors are written before use)
        CoarseWS32& c32 = cws32;
        float* const vs[8] = {c32.wxl, c32.wyl, c32.r, c32.w, c32.mw, c32.p, c32.ap, c32.mp};
        for (int i = 0; i < 8; ++i) zero_vec(vs[i], nc);
        zero_mg(c32.mg);
        __syncthreads();
        const double* ac = P.a_c + b * ncT;
        const double* bc = rxn ? P.b_c + b * ncT : nullptr;
        CellCheck cells;
        cells.look(nc, ac, bc);
        operator32(c32, nc, ac, bc, 0);
        if (!cells.finish(red)) flags |= kFlagBadCoef;
        const int ks = scale_of_cells(cells.amax, cells.bmax);
        if (ks != 0) operator32_scaled(c32, nc, ac, bc, ks);  // (coefficients beyond 2^-16 .. 2^15)
        if (cold) {
          const float inc = 1.0f / (float)nc;
          for_interior(nc, [&](int p, int i, int j) {
            c32.xh[p] = sinpif(i * inc) * sinpif(j * inc);
            c32.xl[p] = 0.0f;
          });
        }
        __syncthreads();
        eit = lobpcg32(c32, nc, P.tol_eig, P.max_eig_it, P.nu, omega, red, &esh32, cold ? 20.0 : pow2(-ks) * lam_prev, lamH,
                       gH);
        lam_prev = lamH *= pow2(ks);
        if (eit < 0) flags |= kFlagEigNoConv;
        if (P.u_out) {
          for_interior(nc, [&](int p, int i, int j) {
            P.u_out[b * (size_t)(nc - 1) * (nc - 1) + (j - 1) * (nc - 1) + (i - 1)] = uH[p];
          });
        }
        if (P.u_pad) {
          const size_t Vc = gsz(nc);
          for_all(Vc, [&](size_t q) { P.u_pad[b * Vc + q] = uH[(int)q]; });
        }
        __syncthreads();
      } else {
        // the fine solves of the previous point reused this memory: clear the coarse vectors
        // (rings must be zero; interiors are written before use)
        double* vs[11] = {cw.wx, cw.wy, cw.x, cw.Ax, cw.Mx, cw.w, cw.Aw, cw.Mw, cw.p, cw.Ap, cw.Mp};
        for (int i = 0; i < 11; ++i) zero_vec(vs[i], nc);
        if (rxn) {
          zero_vec(cw.rx, nc);
          zero_vec(cw.ry, nc);
          zero_vec(cw.rd, nc);
        }
        zero_vec(cw.r32, nc);
        zero_vec(cw.w32, nc);
        zero_mg(cw.mg);
        __syncthreads();
        const double* ac = P.a_c + b * ncT;
        const double* bc = rxn ? P.b_c + b * ncT : nullptr;
        CellCheck cells;
        cells.look(nc, ac, bc);
        operator64(cw, nc, ac, bc, 0);
        if (!cells.finish(red)) flags |= kFlagBadCoef;
        const int ks = scale_of_cells(cells.amax, cells.bmax);  // (its V-cycles and Gram matrices are FP32)
        if (ks != 0) operator64_scaled(cw, nc, ac, bc, ks);
        if (cold) {
          const float inc = 1.0f / (float)nc;
          for_interior(nc, [&](int p, int i, int j) { cw.x[p] = (double)(sinpif(i * inc) * sinpif(j * inc)); });
        } else {
          for_interior(nc, [&](int p, int, int) { cw.x[p] = cw.uprev[p]; });
        }
        __syncthreads();
        eit = lobpcg(cw, nc, P.tol_eig, P.max_eig_it, P.nu, omega, red, &esh, lamH, gH);
        lam_prev = lamH *= pow2(ks);
        if (eit < 0) flags |= kFlagEigNoConv;
        for_interior(nc, [&](int p, int, int) { cw.uprev[p] = cw.x[p]; });
        if (P.u_out) {
          for_interior(nc, [&](int p, int i, int j) {
            P.u_out[b * (size_t)(nc - 1) * (nc - 1) + (j - 1) * (nc - 1) + (i - 1)] = cw.x[p];
          });
        }
        if (P.u_pad) {
          const size_t Vc = gsz(nc);
          for_all(Vc, [&](size_t q) { P.u_pad[b * Vc + q] = cw.x[q]; });
        }
        __syncthreads();
      }
      // ---- fine two-grid updates (Algorithm 1 steps 2-4; Algorithm 2 steps 9-14); a solve of
      // mode 2 runs elsewhere and leaves the coarse eigenvalue as a placeholder
      // the quantity of interest of a level whose eigenpair is the coarse one: lambda_H or G(u_H)
      // (the reuse scheme gives coarse pairs only to levels that solve their own fine problems)
      const double qH = P.qoi ? gH : lamH;
      double lf = qH, lp = P.np > 0 ? qH : 0.0;
      double gf = 0.0, gp = 0.0;
      int itf = 0, itp = 0, of = 0, op = 0;
      const double* rbf = rxn ? P.b_f + b * nfT : nullptr;
      const double* rbp = rxn ? P.b_p + b * npT : nullptr;
      if (!P.direct_f) {
        if (P.mode_f != 2) lf = fine(P.nf, P.a_f + b * nfT, rbf, lamH, itf, of, flags, gf);
        if (P.qoi && P.mode_f != 2) lf = gf;
      }
      if (P.prev_given) {
        lp = P.out[b * 4 + 2];  // every thread reads it before thread 0 rewrites the same value below
      } else if (P.np > 0 && !P.direct_p) {
        if (P.mode_p != 2) lp = fine(P.np, P.a_p + b * npT, rbp, lamH, itp, op, flags, gp);
        if (P.qoi && P.mode_p != 2) lp = gp;
      }
      if (threadIdx.x == 0) {
        P.out[b * 4 + 0] = lamH;
        P.out[b * 4 + 1] = lf;
        P.out[b * 4 + 2] = lp;
        P.out[b * 4 + 3] = lf - lp;
        P.stat[b * 4 + 0] = eit < 0 ? P.max_eig_it : eit;
        P.stat[b * 4 + 1] = itf;
        P.stat[b * 4 + 2] = itp;
        P.stat[b * 4 + 3] = flags;
        P.outer[b * 2 + 0] = of;
        P.outer[b * 2 + 1] = op;
      }
    }
  }
}

// Operator application for parity checks of the stencils: one CTA per coefficient field; the
// scratch holds four padded grids per field.  Uses the same weight builders and stencils as the
// solver.  which: 0 stiffness, 1 mass, 2 stiffness - sigma mass; 3 the reaction matrix of the
// field (edge-weight form), 4 the same from the centroid values.
__global__ void apply_kernel(int n, const double* __restrict__ a, int which, double sigma,
                             const double* __restrict__ x, double* __restrict__ y, double* scratch) {
  const size_t V = gsz(n);
  const size_t b = blockIdx.x;
  double* wx = scratch + b * 4 * V;
  double* wy = wx + V;
  double* xp = wy + V;
  double* wd = xp + V;
  const size_t nT = (size_t)2 * n * n, nI = (size_t)(n - 1) * (n - 1);
  const double* ab = a + b * nT;
  if (which == 3)
    reaction_weights<double, double>(n, ab, ab + (size_t)n * n, wx, wy, wd);
  else
    weights_from_cells<double, double>(n, ab, ab + (size_t)n * n, wx, wy);
  for_all(V, [&](size_t q) { xp[q] = 0.0; });
  __syncthreads();
  for_interior(n, [&](int p, int i, int j) { xp[p] = x[b * nI + (size_t)(j - 1) * (n - 1) + (i - 1)]; });
  __syncthreads();
  const int ld = n + 1;
  const double hm = 1.0 / (12.0 * n * n);
  for_interior(n, [&](int p, int i, int j) {
    double v;
    if (which == 3) {
      v = hm * react7<double, double>(wx, wy, wd, xp, p, ld);
    } else if (which == 4) {
      v = hm * react_cells(ab, n, xp, p, ld, i, j);
    } else {
      const double ax = stiff<double, double>(wx, wy, xp, p, ld);
      const double mx = hm * mass7(xp, p, ld);
      v = which == 0 ? ax : which == 1 ? mx : ax - sigma * mx;
    }
    y[b * nI + (size_t)(j - 1) * (n - 1) + (i - 1)] = v;
  });
}

// Per-shift sums of the per-sample differences over the points of a batch: one CTA per shift,
// fixed reduction order (deterministic).  flags receives the OR of all sample flags.
__global__ void shift_sums_kernel(const double* __restrict__ out, const int* __restrict__ stat, int npts,
                                  double* __restrict__ sums, int* __restrict__ flags, int accumulate) {
  __shared__ double red[kRedSlots];
  const int r = blockIdx.x;
  double acc[1] = {0.0}, o[1];
  int f = 0;
  for (int k = threadIdx.x; k < npts; k += blockDim.x) {
    const size_t b = (size_t)r * npts + k;
    acc[0] += out[b * 4 + 3];
    f |= stat[b * 4 + 3];
  }
  block_sum<1, double>(acc, o, red);
  if (f) atomicOr(flags, f);
  if (threadIdx.x == 0) sums[r] = accumulate ? sums[r] + o[0] : o[0];
}

// reuse scheme: gather the stored level-0 pairs (and the level below's values) of a pass's samples
__global__ void reuse_gather_kernel(int R, int npts, uint32_t k0, size_t V, const double* __restrict__ u0,
                                    const double* __restrict__ lam0, uint32_t ld0, const double* __restrict__ lamp,
                                    uint32_t ldp, double* __restrict__ upad, double* __restrict__ out,
                                    const uint32_t* dk) {
  if (dk) k0 += *dk;
  const size_t B = (size_t)R * npts, tot = B * V;
  for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < tot; q += (size_t)gridDim.x * blockDim.x) {
    const size_t b = q / V, e = q % V;
    const size_t r = b / npts, k = k0 + b % npts;
    upad[q] = u0[(r * ld0 + k) * V + e];
    if (e == 0) {
      out[b * 4 + 0] = lam0[r * ld0 + k];
      out[b * 4 + 2] = lamp ? lamp[r * ldp + k] : 0.0;
    }
  }
}

__global__ void reuse_scatter_kernel(int R, int npts, uint32_t k0, size_t V, const double* __restrict__ upad,
                                     const double* __restrict__ out, double* __restrict__ lam, uint32_t ldl,
                                     double* __restrict__ u0, double* __restrict__ lam0, uint32_t ld0,
                                     const uint32_t* dk) {
  if (dk) k0 += *dk;
  const size_t B = (size_t)R * npts, tot = B * (u0 ? V : 1);
  const size_t per = u0 ? V : 1;
  for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < tot; q += (size_t)gridDim.x * blockDim.x) {
    const size_t b = q / per, e = q % per;
    const size_t r = b / npts, k = k0 + b % npts;
    if (u0) u0[(r * ld0 + k) * V + e] = upad[q];
    if (e == 0) {
      lam[r * ldl + k] = out[b * 4 + 1];
      if (lam0) lam0[r * ld0 + k] = out[b * 4 + 0];
    }
  }
}

int grid_of(size_t n) {
  size_t g = (n + 255) / 256;
  return (int)(g < 1 ? 1 : (g > 152 * 32 ? 152 * 32 : g));
}

}  // namespace

cudaError_t launch_reuse_gather(int R, int npts, uint32_t k0, size_t V, const double* d_u0, const double* d_lam0,
                                uint32_t ld0, const double* d_lamp, uint32_t ldp, double* d_upad, double* d_out,
                                cudaStream_t st, const uint32_t* d_kshift) {
  const size_t tot = (size_t)R * npts * V;
  if (tot == 0) return cudaSuccess;
  reuse_gather_kernel<<<grid_of(tot), 256, 0, st>>>(R, npts, k0, V, d_u0, d_lam0, ld0, d_lamp, ldp, d_upad, d_out,
                                                    d_kshift);
  return cudaGetLastError();
}

cudaError_t launch_reuse_scatter(int R, int npts, uint32_t k0, size_t V, const double* d_upad, const double* d_out,
                                 double* d_lam, uint32_t ldl, double* d_u0, double* d_lam0, uint32_t ld0,
                                 cudaStream_t st, const uint32_t* d_kshift) {
  const size_t tot = (size_t)R * npts * (d_u0 ? V : 1);
  if (tot == 0) return cudaSuccess;
  reuse_scatter_kernel<<<grid_of(tot), 256, 0, st>>>(R, npts, k0, V, d_upad, d_out, d_lam, ldl, d_u0, d_lam0, ld0,
                                                     d_kshift);
  return cudaGetLastError();
}

size_t sample_fallback_bytes(int n, int reaction) {
  Carver c(nullptr);
  c.take<FineWS<double>>(1);
  c.take<MinresShared<double>>(1);
  c.take<double2>(1);
  return (c.used() + fine_bytes<double>(n, reaction != 0) + 255) & ~(size_t)255;
}

size_t sample_slab_bytes(int nf, int nc, int np, int mixed, int eig32, int mode_f, int mode_p, int reaction) {
  return mixed ? slab_size<float>(nf, nc, np, eig32 != 0, mode_f, mode_p, reaction != 0)
               : slab_size<double>(nf, nc, np, false, mode_f, mode_p, reaction != 0);
}

namespace {
using SampleFn = void (*)(SampleLaunch);
SampleFn sample_fn(int mixed, int threads, int wide) {
  return mixed ? (threads <= 256 && !wide ? sample_kernel<float, 256> : sample_kernel<float, 512>) : sample_kernel<double, 512>;
}
}  // namespace

int sample_occupancy(int mixed, int threads, size_t smem, int wide) {
  int nb = 0;
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, sample_fn(mixed, threads, wide), threads, smem);
  return e == cudaSuccess ? nb : 0;
}

int sample_static_smem(int mixed) {
  cudaFuncAttributes fa;
  const cudaError_t e = cudaFuncGetAttributes(&fa, sample_fn(mixed, 512, 1));
  return e == cudaSuccess ? (int)fa.sharedSizeBytes : 8192;
}

cudaError_t raise_smem_limit(const void* func, int bytes) {
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, int> limit;  // (device, kernel) -> limit set so far
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  int& cur = limit[{dev, func}];
  if (bytes <= cur) return cudaSuccess;
  e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) cur = bytes;
  return e;
}

cudaError_t set_sample_smem(int mixed, int bytes) {
  const cudaError_t e = raise_smem_limit((const void*)sample_fn(mixed, 256, 0), bytes);
  return e == cudaSuccess ? raise_smem_limit((const void*)sample_fn(mixed, 512, 1), bytes) : e;
}

cudaError_t launch_apply_operator(int n, int B, const double* d_a, int which, double sigma, const double* d_x,
                                  double* d_y, double* d_scratch, cudaStream_t st) {
  if (B == 0) return cudaSuccess;
  apply_kernel<<<B, 256, 0, st>>>(n, d_a, which, sigma, d_x, d_y, d_scratch);
  return cudaGetLastError();
}

cudaError_t launch_shift_sums(const double* d_out, const int* d_stat, int R, int npts, double* d_sums, int* d_flags,
                              cudaStream_t st, int accumulate) {
  if (R == 0) return cudaSuccess;
  shift_sums_kernel<<<R, 256, 0, st>>>(d_out, d_stat, npts, d_sums, d_flags, accumulate);
  return cudaGetLastError();
}

cudaError_t launch_sample(const SampleLaunch& p, int mixed, int blocks, int threads, size_t smem, cudaStream_t st,
                          int wide) {
  sample_fn(mixed, threads, wide)<<<blocks, threads, smem, st>>>(p);
  return cudaGetLastError();
}

}  // namespace mq

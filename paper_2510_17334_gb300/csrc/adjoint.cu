// Adjoint of the eigenpairs with respect to the values of A and B on their pattern.
//
// For a simple eigenpair (lambda, x) of A x = lambda B x with x^T B x = 1, first-order
// perturbation gives d lambda = x^T (dA - lambda dB) x.  Treating every stored entry
// e = (r_e, c_e) as an independent parameter, a loss with gradient g_lambda[i] has
//   dL/dA_e = sum_i g_i x_i[r_e] x_i[c_e],   dL/dB_e = -sum_i g_i lambda_i x_i[r_e] x_i[c_e],
// a sampled dense-dense product (SDDMM) on the pattern.
#include <cuda_runtime.h>

#include <algorithm>

#include "../../include/slrf.h"
#include "common.cuh"
#include "dense.cuh"

namespace slrf {

// The product is bound by GB300's FP64 pipe (2 FMA per clock and SM: a warp instruction takes
// 16 clocks of its SM), so every FP64 operation that is not one of the two FMAs per stored entry
// and eigenpair is kept out of it:
//   * a lane owns a stored entry and runs over the eigenpairs, so nothing is reduced across
//     lanes (a warp reduction of both sums costs 10 FP64 adds an entry, more than the FMAs at
//     k <= 64);
//   * a warp takes the entries of R consecutive rows 32 at a time through a queue, so the lanes
//     stay busy also where rows hold 27 or 81 entries; the row weights sit in shared memory,
//     [eigenpair][row], one 16-byte read per lane and eigenpair;
//   * SYM: the gradient of a symmetric sum sum_i g_i x_i x_i^T is symmetric, so only the entries
//     with column >= row are summed; a second, copying kernel finds the mirror of every other
//     entry by bisection (and sums it directly where the pattern has no mirror).
// 48^3 elasticity box (n = 324,864, 25.2M entries), k = 50: 2.97 ms (25.4 ms with a warp per row,
// lanes over the eigenpairs and a reduction per entry); the FMAs alone take 4.4 ms for every
// entry, 2.2 ms for half of them.
constexpr int kSdWarps = 8;

// Weights of row r for eigenpair i: (g_i x_i, g_i lambda_i x_i) from the eigenvectors, or the
// rows of two given blocks.
struct SdWeights {
  const double *evals, *g;  // SYM: eigenvalues and their gradients
  const double *YA, *YB;    // otherwise: n x k blocks (leading dimension k)
};
template <bool SYM>
__device__ __forceinline__ double2 sd_weight(const SdWeights &w, const double *X, int ldx, int k, int64_t r, int i) {
  if constexpr (SYM) {
    const double x = X[r * ldx + i], g = w.g[i];
    return make_double2(g * x, g * w.evals[i] * x);
  } else {
    return make_double2(w.YA[r * k + i], w.YB[r * k + i]);
  }
}

// V2: the rows of X start on 16-byte boundaries (two eigenpairs per load).
template <bool SYM, bool V2>
__global__ void __launch_bounds__(32 * kSdWarps) sddmm_kernel(int64_t n, const int64_t *__restrict__ rowptr,
                                                              const int32_t *__restrict__ col, int k, int R,
                                                              const double *__restrict__ X, int ldx,
                                                              const SdWeights w, double *__restrict__ gA,
                                                              double *__restrict__ gB) {
  extern __shared__ __align__(16) double2 sd_smem[];  // [warp][k][R]
  __shared__ int64_t q_e[kSdWarps][64];
  __shared__ int q_c[kSdWarps][64];
  __shared__ unsigned char q_s[kSdWarps][64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t r0 = ((int64_t)blockIdx.x * kSdWarps + warp) * R;
  if (r0 >= n) return;  // warp-uniform; only warp-level synchronisation below
  const int rows = (int)(n - r0 < R ? n - r0 : R);
  double2 *const ws = sd_smem + (size_t)warp * k * R;
  for (int s = 0; s < rows; ++s)
    for (int i = lane; i < k; i += 32) ws[i * R + s] = sd_weight<SYM>(w, X, ldx, k, r0 + s, i);
  const int64_t e0 = rowptr[r0], e1 = rowptr[r0 + rows];
  const int64_t my_end = rowptr[r0 + (lane < rows ? lane + 1 : rows)];  // lane s: end of row s
  int64_t *const qe = q_e[warp];
  int *const qc = q_c[warp];
  unsigned char *const qs = q_s[warp];
  __syncwarp();
  // the first m (<= 32) queued entries, one per lane
  auto process = [&](int m) {
    if (lane < m) {
      const int64_t e = qe[lane];
      const double *xc = X + (int64_t)qc[lane] * ldx;
      const double2 *wr = ws + qs[lane];
      double sa0 = 0.0, sb0 = 0.0, sa1 = 0.0, sb1 = 0.0;
      int i = 0;
      if constexpr (V2) {
#pragma unroll 4
        for (; i + 2 <= k; i += 2) {
          const double2 x = *reinterpret_cast<const double2 *>(xc + i);
          const double2 w0 = wr[i * R], w1 = wr[(i + 1) * R];
          sa0 = fma(w0.x, x.x, sa0);
          sb0 = fma(w0.y, x.x, sb0);
          sa1 = fma(w1.x, x.y, sa1);
          sb1 = fma(w1.y, x.y, sb1);
        }
      } else {
#pragma unroll 4
        for (; i + 2 <= k; i += 2) {
          const double x0 = xc[i], x1 = xc[i + 1];
          const double2 w0 = wr[i * R], w1 = wr[(i + 1) * R];
          sa0 = fma(w0.x, x0, sa0);
          sb0 = fma(w0.y, x0, sb0);
          sa1 = fma(w1.x, x1, sa1);
          sb1 = fma(w1.y, x1, sb1);
        }
      }
      if (i < k) {
        const double x = xc[i];
        const double2 w0 = wr[i * R];
        sa0 = fma(w0.x, x, sa0);
        sb0 = fma(w0.y, x, sb0);
      }
      gA[e] = sa0 + sa1;
      gB[e] = -(sb0 + sb1);
    }
    __syncwarp();
  };
  int nq = 0;
  for (int64_t base = e0; base < e1; base += 32) {
    const int64_t e = base + lane;
    int s = 0;
    for (int t = 0; t + 1 < rows; ++t) s += e >= __shfl_sync(0xffffffffu, my_end, t) ? 1 : 0;
    const int c = e < e1 ? col[e] : 0;
    const bool take = e < e1 && (!SYM || c >= r0 + s);
    const unsigned mask = __ballot_sync(0xffffffffu, take);
    if (take) {
      const int at = nq + __popc(mask & ((1u << lane) - 1u));
      qe[at] = e;
      qc[at] = c;
      qs[at] = (unsigned char)s;
    }
    nq += __popc(mask);
    __syncwarp();
    if (nq >= 32) {
      process(32);
      nq -= 32;
      if (lane < nq) {  // the rest moves to the front (source and target do not overlap)
        qe[lane] = qe[32 + lane];
        qc[lane] = qc[32 + lane];
        qs[lane] = qs[32 + lane];
      }
      __syncwarp();
    }
  }
  process(nq);
}

// The entries with column < row of a symmetric product: copied from their mirror, found by
// bisection in row c; an entry without one (or in an unsorted row) is summed here.
__global__ void __launch_bounds__(256) sddmm_mirror_kernel(int64_t n, const int64_t *__restrict__ rowptr,
                                                           const int32_t *__restrict__ col, int k,
                                                           const double *__restrict__ X, int ldx, const SdWeights w,
                                                           double *gA, double *gB) {
  const int lane = threadIdx.x & 31;
  const int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (r >= n) return;
  const int64_t e1 = rowptr[r + 1];
  for (int64_t e = rowptr[r] + lane; e < e1; e += 32) {
    const int c = col[e];
    if (c >= r) continue;
    int64_t lo = rowptr[c];
    const int64_t end = rowptr[c + 1];
    int64_t hi = end;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (col[mid] < r) lo = mid + 1;
      else hi = mid;
    }
    if (lo < end && col[lo] == r) {
      gA[e] = gA[lo];
      gB[e] = gB[lo];
      continue;
    }
    double sa = 0.0, sb = 0.0;
    for (int i = 0; i < k; ++i) {
      const double2 wi = sd_weight<true>(w, X, ldx, k, r, i);
      const double x = X[(int64_t)c * ldx + i];
      sa = fma(wi.x, x, sa);
      sb = fma(wi.y, x, sb);
    }
    gA[e] = sa;
    gB[e] = -sb;
  }
}

template <bool SYM>
static int sddmm(int64_t n, const int64_t *rowptr, const int32_t *col, int k, const double *X, int ldx,
                 const SdWeights &w, double *gA, double *gB, cudaStream_t st) {
  const size_t per_row = kSdWarps * (size_t)k * sizeof(double2);  // shared memory of one row per warp
  if (per_row > 200 * 1024) return SLRF_EINVAL;
  // rows per warp: up to 8, within 56 KB a block (4 blocks of 8 warps a SM)
  const int R = (int)std::max<size_t>(1, std::min<size_t>(8, (56 * 1024) / per_row));
  const size_t smem = per_row * R;
  const bool v2 = ldx % 2 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
  const auto kernel = v2 ? sddmm_kernel<SYM, true> : sddmm_kernel<SYM, false>;
  if (smem > 48 * 1024 &&
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) != cudaSuccess)
    return SLRF_ECUDA;
  const int64_t per_block = (int64_t)kSdWarps * R;
  kernel<<<(unsigned)((n + per_block - 1) / per_block), 32 * kSdWarps, smem, st>>>(n, rowptr, col, k, R, X, ldx, w, gA,
                                                                                  gB);
  if (SYM)
    sddmm_mirror_kernel<<<(unsigned)((n + 7) / 8), 256, 0, st>>>(n, rowptr, col, k, X, ldx, w, gA, gB);
  return cudaGetLastError() == cudaSuccess ? SLRF_OK : SLRF_ECUDA;
}

int eig_grad_values(int64_t n, const int64_t *rowptr, const int32_t *col, int k, const double *evals,
                    const double *X, int ldx, const double *g, double *gA, double *gB, cudaStream_t st) {
  return sddmm<true>(n, rowptr, col, k, X, ldx, SdWeights{evals, g, nullptr, nullptr}, gA, gB, st);
}

}  // namespace slrf

// ============================================================================== a13
// Eigenvector terms of the adjoint.  For each eigenpair i (columns of n x k row-major
// blocks, leading dimension k) solve the singular, consistent symmetric system
//   (A - lambda_i B) xi_i = b_i,   b_i = -(g_x_i - B x_i (x_i^T g_x_i))   (b_i orthogonal to x_i)
// by MINRES (Paige & Saunders, 1975) on all columns at once, then make xi_i B-orthogonal
// to x_i.  Per column the Lanczos/Givens scalars live on the device; every column keeps
// iterating until its residual estimate phibar <= tol * ||b_i|| or the cap.
namespace slrf {

struct MinresScal {
  double beta, oldb, dbar, epsln, phibar, cs, sn, alfa, beta1;
  double oldeps, delta, gamma, phi;
  int active, iters;
};

constexpr int kAdjRows = 512;

// partial column sums of x .* y over row chunks: work[chunk][k]
__global__ void colprod_partial_kernel(int64_t n, int k, const double *x, const double *y, double *work) {
  const int c = blockIdx.y * blockDim.x + threadIdx.x;
  if (c >= k) return;
  const int64_t r0 = (int64_t)blockIdx.x * kAdjRows;
  const int64_t r1 = r0 + kAdjRows < n ? r0 + kAdjRows : n;
  double s = 0.0;
  for (int64_t i = r0; i < r1; ++i) s = fma(x[i * k + c], y[i * k + c], s);
  work[(size_t)blockIdx.x * k + c] = s;
}
static void colprod(int64_t n, int k, const double *x, const double *y, double *work, cudaStream_t st) {
  dim3 g((unsigned)((n + kAdjRows - 1) / kAdjRows), (k + 127) / 128);
  colprod_partial_kernel<<<g, 128, 0, st>>>(n, k, x, y, work);
}
__device__ __forceinline__ double colprod_final(const double *work, int nch, int k, int c) {
  double s = 0.0;
  for (int z = 0; z < nch; ++z) s += work[(size_t)z * k + c];
  return s;
}

// b = -(g - Bx (x^T g)); x^T g from partials
__global__ void adj_rhs_kernel(int64_t n, int k, const double *g, const double *BX, const double *work, int nch,
                               double *b) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * k) return;
  const int c = (int)(t % k);
  const double xg = colprod_final(work, nch, k, c);
  b[t] = -(g[t] - BX[t] * xg);
}

// init per column: beta1 = ||b||, r1 = r2 = y = b, x = w = w2 = 0
__global__ void minres_init_scal_kernel(int k, const double *work, int nch, MinresScal *s) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= k) return;
  const double b2 = colprod_final(work, nch, k, c);
  MinresScal m{};
  m.beta1 = sqrt(b2);
  m.beta = m.beta1;
  m.oldb = 0.0;
  m.dbar = 0.0;
  m.epsln = 0.0;
  m.phibar = m.beta1;
  m.cs = -1.0;
  m.sn = 0.0;
  m.active = m.beta1 > 0.0 ? 1 : 0;
  m.iters = 0;
  s[c] = m;
}

// v = y / beta (beta of this step), y = A v - lambda B v - (beta / oldb) r1  [with AV, BV of v]
__global__ void minres_v_kernel(int64_t n, int k, const double *y, const MinresScal *s, double *v) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * k) return;
  const int c = (int)(t % k);
  const MinresScal &m = s[c];
  v[t] = (m.active && m.beta > 0.0) ? y[t] / m.beta : 0.0;
}
__global__ void minres_apply_kernel(int64_t n, int k, const double *AV, const double *BV, const double *lam,
                                    const double *r1, const MinresScal *s, double *y) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * k) return;
  const int c = (int)(t % k);
  const MinresScal &m = s[c];
  double val = fma(-lam[c], BV[t], AV[t]);
  if (m.oldb > 0.0) val -= (m.beta / m.oldb) * r1[t];
  y[t] = val;
}
// alfa = v^T y (final of partials) stored per column
__global__ void minres_alfa_kernel(int k, const double *work, int nch, MinresScal *s) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= k) return;
  s[c].alfa = colprod_final(work, nch, k, c);
}
// y -= (alfa/beta) r2; r1 = r2; r2 = y
__global__ void minres_y2_kernel(int64_t n, int k, const MinresScal *s, double *y, double *r1, double *r2) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * k) return;
  const int c = (int)(t % k);
  const MinresScal &m = s[c];
  const double yy = m.beta > 0.0 ? y[t] - (m.alfa / m.beta) * r2[t] : y[t];
  r1[t] = r2[t];
  r2[t] = yy;
  y[t] = yy;
}
// Givens step with beta_new = ||y|| (final of partials); convergence test
__global__ void minres_scal_kernel(int k, const double *work, int nch, double tol, int itn, MinresScal *s) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= k) return;
  MinresScal m = s[c];
  if (!m.active) return;
  const double bnew = sqrt(colprod_final(work, nch, k, c));
  m.oldb = m.beta;
  m.beta = bnew;
  m.oldeps = m.epsln;
  m.delta = m.cs * m.dbar + m.sn * m.alfa;
  const double gbar = m.sn * m.dbar - m.cs * m.alfa;
  m.epsln = m.sn * m.beta;
  m.dbar = -m.cs * m.beta;
  double gam = sqrt(gbar * gbar + m.beta * m.beta);
  if (!(gam > 1e-300)) gam = 1e-300;
  m.gamma = gam;
  m.cs = gbar / gam;
  m.sn = m.beta / gam;
  m.phi = m.cs * m.phibar;
  m.phibar = m.sn * m.phibar;
  m.iters = itn;
  s[c] = m;
}
// w1 = w2; w2 = w; w = (v - oldeps w1 - delta w2)/gamma; x += phi w; then the column stops
// once phibar <= tol beta1 (the state of a stopped column is frozen)
__global__ void minres_w_kernel(int64_t n, int k, const double *v, const MinresScal *s, double *w, double *w2,
                                double *x) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * k) return;
  const int c = (int)(t % k);
  const MinresScal &m = s[c];
  if (!m.active) return;
  const double w1 = w2[t];
  const double wo = w[t];
  const double wn = (v[t] - m.oldeps * w1 - m.delta * wo) / m.gamma;
  w2[t] = wo;
  w[t] = wn;
  x[t] = fma(m.phi, wn, x[t]);
}
__global__ void minres_stop_kernel(int k, double tol, MinresScal *s, int *notconv, int last) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= k) return;
  MinresScal &m = s[c];
  if (m.active && (m.phibar <= tol * m.beta1 || m.beta == 0.0)) m.active = 0;
  if (last && m.active) atomicExch(notconv, 1);
}
__global__ void minres_count_kernel(int k, const MinresScal *s, int *count) {
  int c = 0;
  for (int i = threadIdx.x; i < k; i += blockDim.x) c += s[i].active;
  c = warp_sum(c);
  __shared__ int sh[4];
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) *count = sh[0] + sh[1] + sh[2] + sh[3];
}
// xi -= x (x^T B xi); then YA = X diag(a) + Xi, YB = X diag(b) + Xi diag(lambda)
__global__ void adj_finish_kernel(int64_t n, int k, const double *X, const double *xi, const double *work, int nch,
                                  const double *lam, const double *g_eval, const double *work2, double *YA,
                                  double *YB) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * k) return;
  const int c = (int)(t % k);
  const double xbxi = colprod_final(work, nch, k, c);   // x^T B xi
  const double gx = colprod_final(work2, nch, k, c);    // g_x^T x
  const double xv = X[t];
  const double xiv = xi[t] - xv * xbxi;
  YA[t] = g_eval[c] * xv + xiv;
  YB[t] = (g_eval[c] * lam[c] + 0.5 * gx) * xv + lam[c] * xiv;
}

struct AdjBuffers {
  double *b, *y, *v, *r1, *r2, *w, *w2, *x, *AV, *BV, *YA, *YB, *work, *work2;
  MinresScal *scal;
  int *flag;
};

// The caller (slrf.cu) provides n x k scratch blocks (X here has leading dimension k).
int eig_grad_vectors(int64_t n, const int64_t *rowptr, const int32_t *col, const double *valA, const double *valB,
                     int k, const double *evals, const double *X, const double *g_eval, const double *g_X,
                     double *gA, double *gB, AdjBuffers bf, int maxit, double tol, int *h_active, int *notconv,
                     cudaStream_t st) {
  const int nch = (int)((n + kAdjRows - 1) / kAdjRows);
  const int64_t tot = n * k;
  const unsigned gb = (unsigned)((tot + 255) / 256);
  // right-hand sides
  spmm_real(n, rowptr, col, valA, valB, X, k, k, nullptr, bf.BV, k, st);
  colprod(n, k, X, g_X, bf.work2, st);  // x^T g
  adj_rhs_kernel<<<gb, 256, 0, st>>>(n, k, g_X, bf.BV, bf.work2, nch, bf.b);
  colprod(n, k, bf.b, bf.b, bf.work, st);
  minres_init_scal_kernel<<<(k + 127) / 128, 128, 0, st>>>(k, bf.work, nch, bf.scal);
  cudaMemcpyAsync(bf.y, bf.b, tot * sizeof(double), cudaMemcpyDeviceToDevice, st);
  cudaMemcpyAsync(bf.r1, bf.b, tot * sizeof(double), cudaMemcpyDeviceToDevice, st);
  cudaMemcpyAsync(bf.r2, bf.b, tot * sizeof(double), cudaMemcpyDeviceToDevice, st);
  cudaMemsetAsync(bf.x, 0, tot * sizeof(double), st);
  cudaMemsetAsync(bf.w, 0, tot * sizeof(double), st);
  cudaMemsetAsync(bf.w2, 0, tot * sizeof(double), st);
  cudaMemsetAsync(bf.flag, 0, 2 * sizeof(int), st);
  *notconv = 0;
  int itn = 0;
  while (itn < maxit) {
    const int chunk = maxit - itn < 64 ? maxit - itn : 64;
    for (int j = 0; j < chunk; ++j) {
      ++itn;
      minres_v_kernel<<<gb, 256, 0, st>>>(n, k, bf.y, bf.scal, bf.v);
      spmm_real(n, rowptr, col, valA, valB, bf.v, k, k, bf.AV, bf.BV, k, st);
      minres_apply_kernel<<<gb, 256, 0, st>>>(n, k, bf.AV, bf.BV, evals, bf.r1, bf.scal, bf.y);
      colprod(n, k, bf.v, bf.y, bf.work, st);
      minres_alfa_kernel<<<(k + 127) / 128, 128, 0, st>>>(k, bf.work, nch, bf.scal);
      minres_y2_kernel<<<gb, 256, 0, st>>>(n, k, bf.scal, bf.y, bf.r1, bf.r2);
      colprod(n, k, bf.y, bf.y, bf.work, st);
      minres_scal_kernel<<<(k + 127) / 128, 128, 0, st>>>(k, bf.work, nch, tol, itn, bf.scal);
      minres_w_kernel<<<gb, 256, 0, st>>>(n, k, bf.v, bf.scal, bf.w, bf.w2, bf.x);
      minres_stop_kernel<<<(k + 127) / 128, 128, 0, st>>>(k, tol, bf.scal, bf.flag, itn == maxit);
    }
    // how many columns still iterate: stop early when none
    minres_count_kernel<<<1, 128, 0, st>>>(k, bf.scal, bf.flag + 1);
    if (cudaMemcpyAsync(h_active, bf.flag + 1, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return SLRF_ECUDA;
    if (*h_active == 0) break;
  }
  if (maxit > 0 && itn >= maxit && *h_active > 0) *notconv = 1;
  // B-orthogonal projection, then the pattern gradients
  spmm_real(n, rowptr, col, valA, valB, bf.x, k, k, nullptr, bf.BV, k, st);
  colprod(n, k, X, bf.BV, bf.work, st);  // x^T B xi
  adj_finish_kernel<<<gb, 256, 0, st>>>(n, k, X, bf.x, bf.work, nch, evals, g_eval, bf.work2, bf.YA, bf.YB);
  // gA[e] = sum_i YA[r][i] X[c][i], gB[e] = -sum_i YB[r][i] X[c][i]
  return sddmm<false>(n, rowptr, col, k, X, k, SdWeights{nullptr, nullptr, bf.YA, bf.YB}, gA, gB, st);
}

size_t adj_work_doubles(int64_t n, int k) { return (size_t)((n + kAdjRows - 1) / kAdjRows) * k; }

}  // namespace slrf

// Adjoint of the eigenpairs with respect to the values of A and B on their pattern.
//
// For a simple eigenpair (lambda, x) of A x = lambda B x with x^T B x = 1, first-order
// perturbation gives d lambda = x^T (dA - lambda dB) x.  Treating every stored entry
// e = (r_e, c_e) as an independent parameter, a loss with gradient g_lambda[i] has
//   dL/dA_e = sum_i g_i x_i[r_e] x_i[c_e],   dL/dB_e = -sum_i g_i lambda_i x_i[r_e] x_i[c_e],
// a sampled dense-dense product (SDDMM) on the pattern.
#include <cuda_runtime.h>

#include <algorithm>
#include <utility>

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
  // rows per warp: up to 8, within 56 KB a block; with the 6.5 KB of queues and the 1 KB that the
  // system keeps of each block three blocks of 8 warps share an SM (k = 50: 51,200 B)
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
  double beta, ib, oldb, dbar, epsln, phibar, cs, sn, beta1;  // ib = 1 / beta
  double iob, oldeps, delta, ig, phi;  // of the pending w and x update: 1 / oldb, ..., 1 / gamma
  int active;   // 1 while the column still iterates
  int pending;  // 1: the w and x update of the last step is still to come
};

// All steps between two looks at the convergence run in one cooperative launch
// (minres_loop_kernel); a step is an apply phase (product with the Lanczos vector, first half of
// the recurrence, alfa) and an update phase (second half, beta, Givens step, stopping test), with
// a grid barrier per 32-column tile after each.  The blocks write partial column sums and every
// block adds them itself in the same order, so nothing else is exchanged.  The Lanczos vectors
// rotate through three buffers (no copies), v = r2 / beta is never stored (A v = (A r2) / beta),
// and the w and x update of a step, which needs only the row's own entries, rides on the next
// step's apply.  n = 2,002, k = 16, about 300 steps: the whole adjoint took 96.1 ms with 11 launches a
// step and column sums of 512 rows on a thread, 9.9 ms with two launches a step, now 5.9 ms, 18 to
// 19 us a step (two barriers, the latency of the gathers and of the FP64 roots).
constexpr int kAdjWarps = 8;

// Sum v over the warps of the block and then over the blocks of the tile (gridDim.x of them):
// true in every thread of the last block, where out is the column's sum in lane c of warp 0.
__device__ bool tile_reduce(double v, int k, double *part, unsigned *counter, double &out) {
  __shared__ double sm[kAdjWarps][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = blockIdx.y * 32 + lane;
  sm[warp][lane] = v;
  __syncthreads();
  if (warp == 0 && c < k) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kAdjWarps; ++w) s += sm[w][lane];
    part[(size_t)blockIdx.x * k + c] = s;
  }
  if (!last_block_arrive(counter + blockIdx.y, gridDim.x)) return false;
  double s = 0.0;
  if (c < k) {
#pragma unroll 8
    for (unsigned b = warp; b < gridDim.x; b += kAdjWarps) s += __ldcg(part + (size_t)b * k + c);
  }
  sm[warp][lane] = s;
  __syncthreads();
  out = 0.0;
#pragma unroll
  for (int w = 0; w < kAdjWarps; ++w) out += sm[w][lane];
  if (threadIdx.x == 0) counter[blockIdx.y] = 0u;
  return true;
}

// out[c] = sum over rows of x[:, c] y[:, c]
__global__ void __launch_bounds__(32 * kAdjWarps) colprod_kernel(int64_t n, int k, int rows, const double *x,
                                                                 const double *y, double *part, unsigned *counters,
                                                                 double *out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = blockIdx.y * 32 + lane;
  const int64_t i0 = (int64_t)blockIdx.x * rows, i1 = i0 + rows < n ? i0 + rows : n;
  double s = 0.0, tot;
  if (c < k)
    for (int64_t i = i0 + warp; i < i1; i += kAdjWarps) s = fma(x[i * k + c], y[i * k + c], s);
  if (tile_reduce(s, k, part, counters, tot) && warp == 0 && c < k) out[c] = tot;
}

// b = -(g - Bx (x^T g))
__global__ void adj_rhs_kernel(int64_t n, int k, const double *g, const double *BX, const double *xg, double *b) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * k) return;
  b[t] = -(g[t] - BX[t] * xg[t % k]);
}

// init per column: beta1 = ||b|| (r2 = b, x = w = w2 = 0)
__global__ void minres_init_kernel(int k, const double *b2, MinresScal *s) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= k) return;
  MinresScal m{};
  m.beta1 = sqrt(b2[c]);
  m.beta = m.beta1;
  m.ib = m.beta1 > 0.0 ? 1.0 / m.beta1 : 0.0;
  m.phibar = m.beta1;
  m.cs = -1.0;
  m.active = m.beta1 > 0.0 ? 1 : 0;
  s[c] = m;
}

struct MinresArgs {
  int64_t n;
  int k, rows;  // rows per block
  const int64_t *rowptr;
  const int32_t *col;
  const double *valA, *valB, *lam;
  double *r1, *r2;  // Lanczos vectors of the last two steps (unscaled; beta = ||r2||)
  double *y;        // the next one
  double *w, *w2, *x;
  MinresScal *s;
  double *part;        // two sets of [blocks][k] partial sums
  unsigned *counters;  // one per tile
  int *err;
  double tol;
  int steps, cw;  // steps of this launch (0: only the pending updates); lanes per column group
};

// Sum over the blocks of the tile of their partial sums, the same in every block; scratch
// [kAdjWarps][32].  Result in every warp's lane c.
__device__ __forceinline__ double tile_sum(const double *part, int k, double (*sm)[32]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = blockIdx.y * 32 + lane;
  double s = 0.0;
  if (c < k) {
#pragma unroll 8
    for (unsigned b = warp; b < gridDim.x; b += kAdjWarps) s += __ldcg(part + (size_t)b * k + c);
  }
  __syncthreads();
  sm[warp][lane] = s;
  __syncthreads();
  s = 0.0;
#pragma unroll
  for (int w = 0; w < kAdjWarps; ++w) s += sm[w][lane];
  return s;
}
// This block's partial sum of v over its warps.
__device__ __forceinline__ void block_part(double v, double *part, int k, double (*sm)[32]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = blockIdx.y * 32 + lane;
  __syncthreads();
  sm[warp][lane] = v;
  __syncthreads();
  if (warp == 0 && c < k) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kAdjWarps; ++w) s += sm[w][lane];
    part[(size_t)blockIdx.x * k + c] = s;
  }
}

// A warp takes a row at a time, cw lanes (8, 16 or 32) over the columns of the tile; with
// fewer than 32 columns the 32 / cw lane groups share the row's entries.  A row's own entries
// are always read and written by the same thread; only the gathered rows of r2 come from other
// blocks, after the barrier's acquire.
__global__ void __launch_bounds__(32 * kAdjWarps) minres_loop_kernel(const MinresArgs a) {
  __shared__ double2 s_ab[kAdjWarps][32];
  __shared__ int s_c[kAdjWarps][32];
  __shared__ double sm[kAdjWarps][32];
  __shared__ MinresScal sc[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int sub = lane & (a.cw - 1), group = lane / a.cw, groups = 32 / a.cw;
  const int c = blockIdx.y * 32 + sub;
  const bool ok = c < a.k, own = group == 0;
  const int cl = blockIdx.y * 32 + lane;  // this lane's column where all lanes take columns
  if (warp == 0) sc[lane] = cl < a.k ? a.s[cl] : MinresScal{};
  __syncthreads();
  double *r1 = a.r1, *r2 = a.r2, *y = a.y, *w = a.w, *w2 = a.w2;
  double *const partA = a.part, *const partB = a.part + (size_t)gridDim.x * a.k;
  const double lam = ok ? a.lam[c] : 0.0;
  const unsigned row_bytes = (unsigned)a.k * (unsigned)sizeof(double);
  const int64_t i0 = (int64_t)blockIdx.x * a.rows, i1 = i0 + a.rows < a.n ? i0 + a.rows : a.n;
  GridBarrier gb{a.counters + blockIdx.y, a.err};
  unsigned epoch = 0;
  for (int step = 0;; ++step) {
    const bool last = step == a.steps;  // past the steps of this launch: nothing more, but with
                                        // steps = 0 the pending updates
    if (last && a.steps > 0) break;
    const MinresScal m = sc[sub];
    const bool act = ok && !last && m.active != 0, pend = ok && m.pending != 0;
    // the same in every block of the tile
    const bool more = __syncthreads_or(act) != 0;
    if (!more && !__syncthreads_or(pend)) break;
    // apply: y = (A r2 - lambda B r2) / beta - (beta / oldb) r1, alfa = v^T y
    const double ratio = m.oldb > 0.0 ? m.beta * m.iob : 0.0;
    const bool any = __any_sync(0xffffffffu, act);
    const char *const xl = reinterpret_cast<const char *>(r2 + (ok ? c : 0));
    double sum = 0.0;
    for (int64_t i = i0 + warp; i < i1; i += kAdjWarps) {
      const int64_t t = i * a.k + c;
      double sa = 0.0, sb = 0.0, o1 = 0.0, o2 = 0.0;
      if (own && ok) {
        if (pend || (act && m.oldb > 0.0)) o1 = r1[t];
        if (act) o2 = r2[t];
      }
      if (any) {
        const int64_t rs = a.rowptr[i], re = a.rowptr[i + 1];
        for (int64_t e0 = rs; e0 < re; e0 += 32) {
          const int cnt = (int)(re - e0 < 32 ? re - e0 : 32);
          __syncwarp();
          if (lane < cnt) {
            s_c[warp][lane] = a.col[e0 + lane];
            s_ab[warp][lane] = make_double2(a.valA[e0 + lane], a.valB[e0 + lane]);
          }
          __syncwarp();
#pragma unroll 4
          for (int q = group; q < cnt; q += groups) {
            const double2 ab = s_ab[warp][q];
            const double x =
                *reinterpret_cast<const double *>(xl + (unsigned long long)(unsigned)s_c[warp][q] * row_bytes);
            sa = fma(ab.x, x, sa);
            sb = fma(ab.y, x, sb);
          }
        }
        for (int o = a.cw; o < 32; o <<= 1) {
          sa += __shfl_xor_sync(0xffffffffu, sa, o);
          sb += __shfl_xor_sync(0xffffffffu, sb, o);
        }
      }
      if (own && ok) {
        if (pend) {  // w_new = (v - oldeps w2 - delta w) / gamma, x += phi w_new (v = r1 / oldb)
          const double wn = fma(-m.delta, w[t], fma(-m.oldeps, w2[t], o1 * m.iob)) * m.ig;
          w2[t] = wn;
          a.x[t] = fma(m.phi, wn, a.x[t]);
        }
        if (act) {
          const double yy = fma(-lam, sb, sa) * m.ib - ratio * o1;
          y[t] = yy;
          sum = fma(o2 * m.ib, yy, sum);
        }
      }
    }
    if (!more) {
      // a block may get here before another one has read a.s: the scalars are written back below,
      // behind a barrier
      if (!grid_sync(gb, gridDim.x, epoch)) return;
      if (warp == 0) sc[lane].pending = 0;
      break;
    }
    block_part(own && ok ? sum : 0.0, partA, a.k, sm);
    if (!grid_sync(gb, gridDim.x, epoch)) return;
    const double alfa = tile_sum(partA, a.k, sm);  // lane c: column c
    // update: y -= (alfa / beta) r2, beta = ||y||
    const MinresScal ml = sc[lane];
    const bool actl = cl < a.k && ml.active != 0;
    const double f = actl ? alfa * ml.ib : 0.0;
    sum = 0.0;
    if (actl) {
#pragma unroll 4
      for (int64_t i = i0 + warp; i < i1; i += kAdjWarps) {
        const int64_t t = i * a.k + cl;
        const double yy = y[t] - f * r2[t];
        y[t] = yy;
        sum = fma(yy, yy, sum);
      }
    }
    block_part(sum, partB, a.k, sm);
    if (!grid_sync(gb, gridDim.x, epoch)) return;
    const double b2 = tile_sum(partB, a.k, sm);
    if (warp == 0) {
      MinresScal g = ml;
      g.pending = 0;
      if (actl) {
        g.oldb = g.beta;
        g.iob = g.ib;
        g.ib = b2 > 0.0 ? rsqrt(b2) : 0.0;
        g.beta = b2 * g.ib;
        g.oldeps = g.epsln;
        g.delta = g.cs * g.dbar + g.sn * alfa;
        const double gbar = g.sn * g.dbar - g.cs * alfa;
        g.epsln = g.sn * g.beta;
        g.dbar = -g.cs * g.beta;
        const double g2 = fma(gbar, gbar, b2);  // gamma^2
        g.ig = g2 > 0.0 ? rsqrt(g2) : 1e300;
        g.cs = gbar * g.ig;
        g.sn = g.beta * g.ig;
        g.phi = g.cs * g.phibar;
        g.phibar = g.sn * g.phibar;
        g.pending = 1;
        if (g.phibar <= a.tol * g.beta1 || g.beta == 0.0) g.active = 0;
      }
      sc[lane] = g;
    }
    __syncthreads();
    double *const yo = r1;
    r1 = r2;
    r2 = y;
    y = yo;
    double *const wo = w2;
    w2 = w;
    w = wo;
  }
  // epoch 0: nothing was done and no barrier passed since the blocks read a.s
  if (epoch > 0 && warp == 0 && blockIdx.x == 0 && cl < a.k) a.s[cl] = sc[lane];
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
__global__ void adj_finish_kernel(int64_t n, int k, const double *X, const double *xi, const double *xbxi,
                                  const double *lam, const double *g_eval, const double *gx, double *YA, double *YB) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * k) return;
  const int c = (int)(t % k);
  const double xv = X[t];
  const double xiv = xi[t] - xv * xbxi[c];  // x^T B xi
  YA[t] = g_eval[c] * xv + xiv;
  YB[t] = (g_eval[c] * lam[c] + 0.5 * gx[c]) * xv + lam[c] * xiv;  // g_x^T x
}

struct AdjBuffers {
  double *b, *y, *r, *w, *w2, *x, *BV, *YA, *YB;  // n x k blocks
  double *work, *work2;                           // k words each
  MinresScal *scal;
  double *part;        // adj_part_doubles(k) words
  unsigned *counters;  // a zeroed word per 32 columns, left zero
  int *flag;
};

// Row blocks of the column sums and of the MINRES loop (all resident at once): 16 rows at least.
static int adj_rows(int64_t n, int blocks) {
  const int64_t r = std::max<int64_t>(16, (n + blocks - 1) / blocks);
  return (int)((r + kAdjWarps - 1) / kAdjWarps * kAdjWarps);
}
// Resident blocks of the loop per tile of 32 columns.
static int minres_blocks(int k) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, minres_loop_kernel, 32 * kAdjWarps, 0) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return std::min(per_sm, 4) * device_sm_count() / ((k + 31) / 32);
}
size_t adj_part_doubles(int k) { return 2 * 4 * (size_t)device_sm_count() * k; }
size_t adj_scal_bytes(int k) { return ((size_t)k * sizeof(MinresScal) + 255) / 256 * 256; }

// The caller (slrf.cu) provides n x k scratch blocks (X here has leading dimension k).
int eig_grad_vectors(int64_t n, const int64_t *rowptr, const int32_t *col, const double *valA, const double *valB,
                     int k, const double *evals, const double *X, const double *g_eval, const double *g_X,
                     double *gA, double *gB, AdjBuffers bf, int maxit, double tol, int *h_active, int *notconv,
                     cudaStream_t st) {
  const int64_t tot = n * k;
  const unsigned gb = (unsigned)((tot + 255) / 256);
  const int blocks = minres_blocks(k);
  if (blocks < 1) return SLRF_ECUDA;
  const int rows = adj_rows(n, blocks);
  const dim3 grid((unsigned)((n + rows - 1) / rows), (unsigned)((k + 31) / 32));
  const int cw = k <= 8 ? 8 : (k <= 16 ? 16 : 32);
  auto colprod = [&](const double *x, const double *y, double *out) {
    colprod_kernel<<<grid, 32 * kAdjWarps, 0, st>>>(n, k, rows, x, y, bf.part, bf.counters, out);
  };
  // right-hand sides
  spmm_real(n, rowptr, col, valA, valB, X, k, k, nullptr, bf.BV, k, st);
  colprod(X, g_X, bf.work2);  // x^T g
  adj_rhs_kernel<<<gb, 256, 0, st>>>(n, k, g_X, bf.BV, bf.work2, bf.b);
  colprod(bf.b, bf.b, bf.work);
  minres_init_kernel<<<(k + 127) / 128, 128, 0, st>>>(k, bf.work, bf.scal);
  cudaMemsetAsync(bf.x, 0, tot * sizeof(double), st);
  cudaMemsetAsync(bf.w, 0, tot * sizeof(double), st);
  cudaMemsetAsync(bf.w2, 0, tot * sizeof(double), st);
  MinresArgs a{n, k, rows, rowptr, col, valA, valB, evals, bf.r, bf.b, bf.y, bf.w, bf.w2, bf.x, bf.scal, bf.part,
               bf.counters, bf.flag, tol, 0, cw};
  cudaMemsetAsync(bf.flag, 0, 2 * sizeof(int), st);
  // one launch of `steps` steps; the barrier counters start and end at zero
  auto run = [&](int steps) {
    a.steps = steps;
    void *args[] = {&a};
    cudaMemsetAsync(bf.counters, 0, grid.y * sizeof(unsigned), st);
    const cudaError_t e =
        cudaLaunchCooperativeKernel((void *)minres_loop_kernel, grid, dim3(32 * kAdjWarps), args, 0, st);
    cudaMemsetAsync(bf.counters, 0, grid.y * sizeof(unsigned), st);
    for (int j = 0; j < steps; ++j) {  // the buffers after a step: r1 = r2, r2 = y, w2 in front
      double *const y = a.r1;
      a.r1 = a.r2;
      a.r2 = a.y;
      a.y = y;
      std::swap(a.w, a.w2);
    }
    return e == cudaSuccess;
  };
  *notconv = 0;
  *h_active = 0;
  int itn = 0;
  while (itn < maxit) {
    const int chunk = maxit - itn < 64 ? maxit - itn : 64;
    itn += chunk;
    if (!run(chunk)) return SLRF_ECUDA;
    // how many columns still iterate: stop early when none
    minres_count_kernel<<<1, 128, 0, st>>>(k, bf.scal, bf.flag + 1);
    int h[2] = {0, 0};
    if (cudaMemcpyAsync(h_active, bf.flag, 2 * sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return SLRF_ECUDA;
    h[0] = h_active[0];
    h[1] = h_active[1];
    *h_active = h[1];
    if (h[0] != 0) return SLRF_ETIMEOUT;  // a bounded barrier gave up
    if (*h_active == 0) break;
  }
  if (maxit > 0 && itn >= maxit && *h_active > 0) *notconv = 1;
  if (!run(0)) return SLRF_ECUDA;  // pending w and x updates
  // B-orthogonal projection, then the pattern gradients
  spmm_real(n, rowptr, col, valA, valB, bf.x, k, k, nullptr, bf.BV, k, st);
  colprod(X, bf.BV, bf.work);  // x^T B xi
  adj_finish_kernel<<<gb, 256, 0, st>>>(n, k, X, bf.x, bf.work, evals, g_eval, bf.work2, bf.YA, bf.YB);
  // gA[e] = sum_i YA[r][i] X[c][i], gB[e] = -sum_i YB[r][i] X[c][i]
  return sddmm<false>(n, rowptr, col, k, X, k, SdWeights{nullptr, nullptr, bf.YA, bf.YB}, gA, gB, st);
}

}  // namespace slrf

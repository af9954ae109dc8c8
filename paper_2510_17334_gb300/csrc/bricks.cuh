// Brick SpMM of the FP32 COCG: s = (A - sigma B) r with the gathered rows staged in shared
// memory (included by cocg.cu).
//
// A brick is a set of row pairs next to each other in the mesh (4 x 4 x 2 rows of a box) and
// the list of the distinct rows of r that its rows couple to.  A block copies those rows'
// segments of a 64-entry column tile (512 bytes each) and the brick's records into shared memory
// by 1-D bulk copies, then its 8 warps walk the pairs' records, reading the gathered rows from
// shared memory.  Two blocks share an SM, one copying while the other multiplies.
//
// What bounds it: gathering a row per CSR entry through L1 keeps only the loads in flight that
// fit a warp's registers, about half of them miss L1, and every entry costs 4 load wavefronts
// for the row and 3 for its (column, a, b).  A brick of 32 rows with 27 entries each stages 144
// rows instead of gathering 864, through the copy engine (a whole brick in flight, no
// registers), and each of its 576 records costs 4 wavefronts for the row, 2 for its four values
// and 1/4 for the row's place, for two rows at once.  The load/store pipe is 60 % busy, the rest
// is the latency of shared memory at 16 warps an SM.  41^3 nodes, 160 columns, 8 poles:
// 1.50 ms per product with plain rows, 1.21 ms with pairs gathered through L1 (grp_walk),
// 0.96 ms here; HBM floor 0.52 ms.  Pairs and not nodes of 3 rows: an elasticity box (192 rows
// of 512 bytes for 648 records) gained 3 % this way over grp_walk.
#pragma once

// Record area of a pair: 16 bytes of values per record (a0, a1, b0, b1), then one byte per
// record, the place of its row in the brick's row list.
inline int brick_pad(int cmax) { return (cmax + 3) / 4 * 4; }
inline int brick_group_bytes(int cmax) { return brick_pad(cmax) * 16 + (cmax + 15) / 16 * 16; }

template <bool FRESH>
__device__ __forceinline__ void cocg_spmm_brick_body(const CocgArgs<float> &a, const int rb, const int tile,
                                                     unsigned char *smem, uint64_t *bar, unsigned &phase) {
  constexpr int VEC = 2;
  using C = float2;
  using V2 = Vec<float, VEC>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tid = threadIdx.x;
  const int w_tile0 = tile * 64, w0 = w_tile0 + 2 * lane;
  float acc[VEC][2] = {};
  C be[VEC], sg[VEC];
  bool any_act = false;
#pragma unroll
  for (int v = 0; v < VEC; ++v) {
    any_act |= a.ws[w0 + v].active != 0;
    be[v] = to_c<float>(a.ws[w0 + v].beta);
    sg[v] = a.sig[(w0 + v) & (a.mp - 1)];
  }
  // the same for every warp of the block: all look at the whole tile
  if (__any_sync(0xffffffffu, any_act)) {
    const Bricks &B = a.bricks;
    const int gs = B.group_bytes;
    unsigned char *const rec = smem + (size_t)B.max_rows * 512;
    const char *const rt = reinterpret_cast<const char *>(a.r + w_tile0);
    const size_t row_bytes = (size_t)a.W * sizeof(C);
    int b = rb;
    int nr = b < B.count ? B.nrows[b] : 0;
    int row = b < B.count && tid < nr ? B.rows[(size_t)b * kBrickRows + tid] : 0;
    while (b < B.count) {
      // every warp has finished with the previous brick (the barrier below): its reads come
      // before the copies
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      if (tid == 0) {
        mbar_expect_tx(bar, (uint32_t)(nr * 512 + kBrickGroups * gs));
        bulk_g2s(rec, B.rec + (size_t)b * kBrickGroups * gs, (uint32_t)(kBrickGroups * gs), bar);
      }
      if (tid < nr) bulk_g2s(smem + tid * 512, rt + (size_t)row * row_bytes, 512, bar);
      // the warp's two pairs and the next brick's row list, meanwhile
      const int4 g2[2] = {B.groups[(size_t)b * kBrickGroups + warp], B.groups[(size_t)b * kBrickGroups + warp + kWarps]};
      const int bn = b + B.blocks;
      const int nrn = bn < B.count ? B.nrows[bn] : 0;
      const int rown = bn < B.count && tid < nrn ? B.rows[(size_t)bn * kBrickRows + tid] : 0;
      const bool ok = mbar_wait(bar, phase, a.err, 1);
      phase ^= 1u;
      if (__syncthreads_or(!ok)) {  // gave up: wait (bounded) for the copies in flight, then leave
        mbar_wait(bar, phase ^ 1u, a.err, 1);
        break;
      }
      const unsigned char *const xs = smem + lane * 16;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int4 g = g2[h];  // first row, rows (0: none), records, place of the first row
        const unsigned char *const base = rec + (size_t)(warp + h * kWarps) * gs;
        const float4 *const val = reinterpret_cast<const float4 *>(base);
        const uint32_t *const at = reinterpret_cast<const uint32_t *>(base + B.pad * 16);
        C sa[2][VEC], sb[2][VEC];
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int v = 0; v < VEC; ++v) sa[q][v] = sb[q][v] = make_float2(0.f, 0.f);
        auto step = [&](int t, uint32_t place) {
          const float4 m = val[t], x = *reinterpret_cast<const float4 *>(xs + place * 512);
          const C z[VEC] = {make_float2(x.x, x.y), make_float2(x.z, x.w)};
#pragma unroll
          for (int v = 0; v < VEC; ++v) {
            sa[0][v] = ffma2(make_float2(m.x, m.x), z[v], sa[0][v]);
            sa[1][v] = ffma2(make_float2(m.y, m.y), z[v], sa[1][v]);
            sb[0][v] = ffma2(make_float2(m.z, m.z), z[v], sb[0][v]);
            sb[1][v] = ffma2(make_float2(m.w, m.w), z[v], sb[1][v]);
          }
        };
        auto steps = [&](int t0, int t1) {  // whole words of places
#pragma unroll 1
          for (int t = t0; t < t1; t += 4) {
            const uint32_t w = at[t >> 2];
#pragma unroll
            for (int u = 0; u < 4; ++u) step(t + u, (w >> (8 * u)) & 255u);
          }
        };
        const int nt = g.z, words = nt & ~3, early = (nt >> 1) & ~3;
        steps(0, early);
        // the rows' own p and q arrive during the second half of the walk
        V2 pv[2], qv[2];
        if (!FRESH) {
#pragma unroll
          for (int q = 0; q < 2; ++q)
            if (q < g.y) {
              const size_t off = (size_t)(g.x + q) * a.W + w0;
              pv[q] = ldv_cs<float, VEC>(a.p + off);
              qv[q] = ldv_cs<float, VEC>(a.q + off);
            }
        }
        steps(early, words);
        if (words < nt) {
          uint32_t w = at[words >> 2];
          for (int t = words; t < nt; ++t, w >>= 8) step(t, w & 255u);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q)
          if (q < g.y) {
            const size_t off = (size_t)(g.x + q) * a.W + w0;
            const float4 rw = *reinterpret_cast<const float4 *>(xs + (g.w + q) * 512);
            const C rv[VEC] = {make_float2(rw.x, rw.y), make_float2(rw.z, rw.w)};
            V2 pn, qn;
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
              const C s = cfms(sg[v], sb[q][v], sa[q][v]);  // A r - sigma B r
              pn.z[v] = FRESH ? rv[v] : cfma(be[v], pv[q].z[v], rv[v]);
              qn.z[v] = FRESH ? s : cfma(be[v], qv[q].z[v], s);
              acc[v][0] += pn.z[v].x * qn.z[v].x - pn.z[v].y * qn.z[v].y;
              acc[v][1] += pn.z[v].x * qn.z[v].y + pn.z[v].y * qn.z[v].x;
            }
            stv_cs<float, VEC>(a.p + off, pn);
            stv_cs<float, VEC>(a.q + off, qn);
          }
      }
      __syncthreads();
      b = bn;
      nr = nrn;
      row = rown;
    }
  }
  // the reduction's scratch is the staging area (no copy is in flight any more)
  __syncthreads();
  spmm_tail<float, VEC, true>(a, acc, w_tile0, rb, tile, a.bricks.blocks, reinterpret_cast<double *>(smem));
}

template <bool FRESH>
__global__ void __launch_bounds__(kThreads, 2) cocg_spmm_brick_kernel(const CocgArgs<float> a) {
  extern __shared__ __align__(128) unsigned char brick_smem[];
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  unsigned phase = 0;
  cocg_spmm_brick_body<FRESH>(a, blockIdx.x, blockIdx.y, brick_smem, &bar, phase);
}

// ------------------------------------------------------------------------------ build
// Columns of the merged rows [r0, r0 + rows), rows <= 2: f(record, column, a, b), one value per
// row (zero where a row lacks the column).
template <typename F>
__device__ __forceinline__ int merge_pair(const int64_t *__restrict__ rowptr, const int32_t *__restrict__ col,
                                          const double *__restrict__ valA, const double *__restrict__ valB, int r0,
                                          int rows, F &&f) {
  int64_t pos[2], end[2];
  for (int j = 0; j < 2; ++j) {
    pos[j] = j < rows ? rowptr[r0 + j] : 0;
    end[j] = j < rows ? rowptr[r0 + j + 1] : 0;
  }
  int t = 0;
  for (;; ++t) {
    int32_t m = INT32_MAX;
    bool any = false;
    for (int j = 0; j < 2; ++j)
      if (pos[j] < end[j]) { any = true; m = min(m, col[pos[j]]); }
    if (!any) break;
    float av[2] = {0.f, 0.f}, bv[2] = {0.f, 0.f};
    for (int j = 0; j < 2; ++j)
      if (pos[j] < end[j] && col[pos[j]] == m) {
        av[j] = (float)valA[pos[j]];
        bv[j] = (float)valB[pos[j]];
        ++pos[j];
      }
    f(t, m, av, bv);
  }
  return t;
}
// Position of column m in the sorted list (its lower bound).
__device__ __forceinline__ int brick_place(const int *list, int n, int m) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (list[mid] < m) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}
// Key of the longest row, the one next to row n / 2 of several (the lower one of two): its length,
// then 2^31 - 1 less the distance, then whether it is not above.  One atomic per block.
__global__ void __launch_bounds__(256) longest_row_kernel(int64_t n, const int64_t *__restrict__ rowptr,
                                                          unsigned long long *key) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long k = 0;
  if (i < n) {
    const int64_t len = rowptr[i + 1] - rowptr[i], d = i - n / 2;
    k = ((unsigned long long)(len < 0xFFFFFFFF ? len : 0xFFFFFFFF) << 32) |
        (unsigned long long)((0x7FFFFFFF - (d < 0 ? -d : d)) << 1 | (d <= 0));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) k = max(k, __shfl_xor_sync(0xffffffffu, k, o));
  __shared__ unsigned long long w[8];
  if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = k;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < 8; ++q) k = max(k, w[q]);
    atomicMax(key, k);
  }
}
// Most records of a pair.
__global__ void brick_count_kernel(int64_t ngroups, const int64_t *__restrict__ rowptr, const int32_t *__restrict__ col,
                                   const double *__restrict__ valA, const double *__restrict__ valB,
                                   const int4 *__restrict__ groups, unsigned long long *most) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ngroups) return;
  const int4 g = groups[t];
  const int c = merge_pair(rowptr, col, valA, valB, g.x, g.y, [](int, int, const float *, const float *) {});
  atomicMax(most, (unsigned long long)c);
}
// One block per brick.  Pairs come as (first row, rows); their distinct columns are merged from
// the CSR rows, the brick's row list is their sorted union, and every record gets its values and
// the place of its row in the list.  *flag is raised where a brick has more rows than kBrickRows,
// a pair more columns than cmax, a row is not sorted, or a pair's own rows are not among its
// columns; stats: staged rows, records, rows of the largest brick.  Without rec only these are
// found.
constexpr int kBrickSort = 2048;  // >= kBrickGroups * cmax (checked by the host)
__global__ void __launch_bounds__(256) brick_build_kernel(const int64_t *__restrict__ rowptr,
                                                          const int32_t *__restrict__ col,
                                                          const double *__restrict__ valA,
                                                          const double *__restrict__ valB, int cmax, int pad, int gs,
                                                          int4 *groups, int *nrows, int *rows, unsigned char *rec,
                                                          int *flag, unsigned long long *stats) {
  __shared__ int list[kBrickSort];
  __shared__ int uniq[kBrickRows];
  __shared__ int cnt[kBrickGroups];
  __shared__ int warp_cnt[8];
  __shared__ int nu, bad;
  const int b = blockIdx.x, tid = threadIdx.x;
  if (tid == 0) nu = bad = 0;
  for (int i = tid; i < kBrickSort; i += blockDim.x) list[i] = INT32_MAX;
  __syncthreads();
  int4 g = make_int4(0, 0, 0, 0);
  if (tid < kBrickGroups) {
    g = groups[(size_t)b * kBrickGroups + tid];
    int prev = -1;
    g.z = merge_pair(rowptr, col, valA, valB, g.x, g.y, [&](int t, int m, const float *, const float *) {
      if (t < cmax && tid * cmax + t < kBrickSort) list[tid * cmax + t] = m;
      if (m <= prev) bad = 1;
      prev = m;
    });
    cnt[tid] = g.z;
    if (g.z > cmax) bad = 1;
  }
  __syncthreads();
  if (bad) {
    if (tid == 0) atomicExch(flag, 1);
    return;
  }
  // bitonic sort, then the distinct columns in order (one thread per run's first element)
  for (int k = 2; k <= kBrickSort; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = tid; i < kBrickSort; i += blockDim.x) {
        const int l = i ^ j;
        if (l > i && ((list[i] > list[l]) == ((i & k) == 0))) {
          const int x = list[i];
          list[i] = list[l];
          list[l] = x;
        }
      }
      __syncthreads();
    }
  for (int base = 0; base < kBrickSort; base += blockDim.x) {
    const int i = base + tid;
    const bool first = list[i] != INT32_MAX && (i == 0 || list[i - 1] != list[i]);
    const unsigned m = __ballot_sync(0xffffffffu, first);
    if ((tid & 31) == 0) warp_cnt[tid >> 5] = __popc(m);
    __syncthreads();
    int o = nu;
    for (int w = 0; w < (tid >> 5); ++w) o += warp_cnt[w];
    o += __popc(m & ((1u << (tid & 31)) - 1u));
    if (first && o < kBrickRows) uniq[o] = list[i];
    __syncthreads();
    if (tid == 0)
      for (int w = 0; w < 8; ++w) nu += warp_cnt[w];
    __syncthreads();
  }
  if (nu > kBrickRows) {
    if (tid == 0) atomicExch(flag, 1);
    return;
  }
  if (tid == 0) {
    nrows[b] = nu;
    unsigned long long r = 0;
    for (int j = 0; j < kBrickGroups; ++j) r += cnt[j];
    atomicAdd(stats, (unsigned long long)nu);
    atomicAdd(stats + 1, r);
    atomicMax(stats + 2, (unsigned long long)nu);
  }
  if (tid < nu) rows[(size_t)b * kBrickRows + tid] = uniq[tid];
  // places of the pair's own rows (one after the other), or no bricks
  if (tid < kBrickGroups && g.y > 0) {
    g.w = brick_place(uniq, nu, g.x);
    for (int j = 0; j < g.y; ++j)
      if (g.w + j >= nu || uniq[g.w + j] != g.x + j) bad = 1;
  }
  __syncthreads();
  if (bad) {
    if (tid == 0) atomicExch(flag, 1);
    return;
  }
  if (rec != nullptr && tid < kBrickGroups) {
    groups[(size_t)b * kBrickGroups + tid] = g;
    unsigned char *const base = rec + ((size_t)b * kBrickGroups + tid) * gs;
    float4 *const val = reinterpret_cast<float4 *>(base);
    unsigned char *const at = base + (size_t)pad * 16;
    merge_pair(rowptr, col, valA, valB, g.x, g.y, [&](int t, int m, const float *av, const float *bv) {
      val[t] = make_float4(av[0], av[1], bv[0], bv[1]);
      at[t] = (unsigned char)brick_place(uniq, nu, m);
    });
  }
}

// HODLR assembly kernels: dense leaves and partial-pivoted ACA of every
// off-diagonal block (Sec. 3.2; "partial-pivoted LU" in the proof of Lemma 1).
#include "fifa_common.cuh"
#include "fifa_launch.h"

// ---------------------------------------------------------------------------
// Leaf assembly: leaves[leaf](a, b) = k(x_a, x_b) + nugget [a == b], padding 0.
// One CTA per leaf.  Kernel entries are evaluated once per unordered pair:
// diagonal tiles over their lower triangle, off-diagonal tiles mirrored through
// a shared-memory tile so both stores stay coalesced.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_leaf_assemble(const HmatDesc* __restrict__ Hd) {
  Hd += blockIdx.y;  // problem of a batched launch (descriptor arrays)
  const int leaf = blockIdx.x;
  const int L = Hd->L, Bm = Hd->Bm, kind = Hd->kind;
  const double kc = Hd->kc, nug = Hd->nugget;
  const int* bnd = Hd->bnd;
  const double* x = Hd->x;
  double* D = Hd->leaves + (size_t)leaf * Bm * Bm;
  const int s = bnd[bnd_off(L) + leaf], e = bnd[bnd_off(L) + leaf + 1], m = e - s;
  __shared__ double xs[FIFA_LEAF_MAX];
  __shared__ double tile[32][33];
  for (int a = threadIdx.x; a < m; a += blockDim.x) xs[a] = x[s + a];
  __syncthreads();
  const int nt = (Bm + 31) / 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
  // diagonal 32 x 32 tiles: entries (a, b) with a >= b only, mirrored (the
  // kernel is symmetric bit for bit: fl(xa - xb) = -fl(xb - xa))
  for (int bd = 0; bd < nt; ++bd) {
    for (int t = threadIdx.x; t < 32 * 33 / 2; t += blockDim.x) {
      int ia = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
      if ((ia + 1) * (ia + 2) / 2 <= t) ++ia;
      if (ia * (ia + 1) / 2 > t) --ia;
      const int ib = t - ia * (ia + 1) / 2;
      const int a = 32 * bd + ia, b = 32 * bd + ib;
      double v = 0.0;
      if (a < m && b < m) {
        v = kern_entry(kind, kc, xs[a], xs[b]);
        if (a == b) v = __dadd_rn(v, nug);
      }
      if (a < Bm && b < Bm) {
        D[(size_t)b * Bm + a] = v;
        D[(size_t)a * Bm + b] = v;
      }
    }
  }
  for (int bj = 0; bj < nt; ++bj) {
    for (int bi = bj + 1; bi < nt; ++bi) {
      // tile rows a in [32 bi, +32), cols b in [32 bj, +32): entry (a, b)
      for (int yy = ty; yy < 32; yy += 8) {
        int a = 32 * bi + tx, b = 32 * bj + yy;
        double v = 0.0;
        if (a < m && b < m) {
          v = kern_entry(kind, kc, xs[a], xs[b]);
          if (a == b) v = __dadd_rn(v, nug);
        }
        if (a < Bm && b < Bm) D[(size_t)b * Bm + a] = v;
        tile[yy][tx] = v;
      }
      __syncthreads();
      // mirror: entry (b, a) for b in tile cols, a in tile rows -> column a, row b
      for (int yy = ty; yy < 32; yy += 8) {
        int b = 32 * bj + tx, a = 32 * bi + yy;
        if (a < Bm && b < Bm) D[(size_t)a * Bm + b] = tile[tx][yy];
      }
      __syncthreads();
    }
  }
}

// ---------------------------------------------------------------------------
// ACA.  The G CTAs of one block split its rows and columns; every CTA takes
// identical pivot decisions from the same reduced data, so only maxima are
// exchanged and the bases do not depend on G.  CL: the CTAs are a thread-block
// cluster of C CTAs on work[blockIdx.x / C] = {level, node, ..} and exchange
// through distributed shared memory; else work[blockIdx.x] = {level, node, g, G}
// and a group of G > 1 meets at bounded-spin barriers.
// The arithmetic (fused multiply-adds acc - U V with l ascending, the row
// scaled by one IEEE reciprocal of the pivot) matches the CPU reference
// operation for operation.
//
// What bounds it: large blocks the FP64 pipe (11-14 operations per kernel entry
// and k multiply-adds); small ones the chain of 2 (r + 1) dependent phases, each
// a load, one entry's operations (64 cycles apiece for a warp) and a reduction.
// So a phase costs one barrier: a CTA keeps its slices of U and V in shared
// memory as far as they fit (ACA_KEEP doubles), the pivot row's U entries come
// in one load, and a reduction is one shuffle tree per warp, one exchange in
// shared memory and a second tree in every warp: n = 500, 15 blocks, 400 us in
// two launches -> 98 in one; 0.94 -> 0.91 ms for the grouped blocks of n = 200000,
// which the FP64 pipe bounds.  KEEP = false keeps nothing and leaves that memory to
// the L1 cache.
// ---------------------------------------------------------------------------
#define ACA_KEEP 5632  // doubles of U and V kept per CTA (four CTAs per SM)

// Candidate of a reduction: |value| as its IEEE bits (-1.0 for none), index and
// sign packed; ties to the lower index.  u: the largest |value| of any entry.
struct AcaBest {
  long long v, u;
  int p;  // 2 index + (value negative)
};
__device__ __forceinline__ AcaBest aca_none() { return {__double_as_longlong(-1.0), __double_as_longlong(-1.0), 0x7fffffff}; }
__device__ __forceinline__ void aca_take(AcaBest& a, const AcaBest& b) {
  if (b.v > a.v || (b.v == a.v && b.p < a.p)) {
    a.v = b.v;
    a.p = b.p;
  }
  if (b.u > a.u) a.u = b.u;
}
template <int FROM>
__device__ __forceinline__ void aca_shuffle(AcaBest& a) {
#pragma unroll
  for (int o = FROM; o > 0; o >>= 1) {
    AcaBest b;
    b.v = __shfl_xor_sync(0xffffffffu, a.v, o);
    b.u = __shfl_xor_sync(0xffffffffu, a.u, o);
    b.p = __shfl_xor_sync(0xffffffffu, a.p, o);
    aca_take(a, b);
  }
}
// The entry's value from its bits and sign.
__device__ __forceinline__ double aca_value(const AcaBest& a) {
  return __longlong_as_double(a.v | ((long long)(a.p & 1) << 63));
}

__device__ __forceinline__ AcaBest aca_remote(const AcaBest* p, int rank) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  unsigned r;
  AcaBest b;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("ld.shared::cluster.s64 %0, [%1];" : "=l"(b.v) : "r"(r) : "memory");
  asm volatile("ld.shared::cluster.s64 %0, [%1 + 8];" : "=l"(b.u) : "r"(r) : "memory");
  asm volatile("ld.shared::cluster.s32 %0, [%1 + 16];" : "=r"(b.p) : "r"(r) : "memory");
  return b;
}

template <bool CL, bool KEEP>
__global__ void __launch_bounds__(256, 4) k_aca(const HmatDesc* __restrict__ Hd, const int4* __restrict__ work, int C,
                                              AcaGroups groups,
                                              ArgMax* __restrict__ part, unsigned int* __restrict__ bar,
                                              int* __restrict__ abort_flag, size_t pstride) {
  // problem of a batched launch: its descriptor, its partials, barriers and
  // abort flag pstride bytes after the previous problem's
  Hd += blockIdx.y;
  part = (ArgMax*)((char*)part + blockIdx.y * pstride);
  bar = (unsigned int*)((char*)bar + blockIdx.y * pstride);
  abort_flag = (int*)((char*)abort_flag + blockIdx.y * pstride);
  int lvl, bi, g, G;
  if (!CL && groups.levels > 0) {  // smaller groups than the work list's: level after level, block after block
    int b = blockIdx.x;
    lvl = 0;
    while (b >= groups.G[lvl] << lvl) b -= groups.G[lvl] << lvl, ++lvl;
    G = groups.G[lvl];
    bi = b / G;
    g = b % G;
  } else {
    const int4 w = work[CL ? blockIdx.x / C : blockIdx.x];
    lvl = w.x, bi = w.y, g = CL ? blockIdx.x % C : w.z, G = CL ? C : w.w;
  }
  const int base = blockIdx.x - g;
  const int64_t n = Hd->n;
  const int cap = Hd->cap, kind = Hd->kind;
  const double kc = Hd->kc, eps = Hd->eps;
  const double* __restrict__ x = Hd->x;
  double* Bs = Hd->bases + (size_t)lvl * cap * n;
  int s, h, e;
  node_range(Hd->bnd, lvl, bi, s, h, e);
  const int m = h - s, p = e - h;
  const int nid = node_id(lvl, bi);
  const int rc = (m + G - 1) / G, cc = (p + G - 1) / G;
  const int r0 = min(m, g * rc), r1 = min(m, g * rc + rc);
  const int c0 = min(p, g * cc), c1 = min(p, g * cc + cc);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  extern __shared__ double keep[];  // steps l < kl: V on [c0, c1), then U on [r0, r1)
  __shared__ int rowp[FIFA_CAP_MAX], colp[FIFA_CAP_MAX];
  __shared__ double piv_row[FIFA_CAP_MAX];  // the pivot row's U entries, then the pivot column's V entries
  __shared__ AcaBest wbest[2][8], cbest[2];
  const int kl = KEEP ? min(cap, ACA_KEEP / (rc + cc)) : 0, kstep = rc + cc;
  unsigned int phase = 0;

  // reduce over the node's CTAs; two buffers in turn, each written again only
  // after a barrier that follows every read of it
  bool dead = false;
  auto reduce = [&](AcaBest a) -> AcaBest {
    aca_shuffle<16>(a);
    AcaBest* wb = wbest[phase & 1u];
    if (lane == 0) wb[warp] = a;
    __syncthreads();
    a = wb[lane & 7];
    aca_shuffle<4>(a);
    if (G > 1) {
      if constexpr (CL) {
        if (tid == 0) cbest[phase & 1u] = a;
        cluster_sync_all();
        a = aca_remote(&cbest[phase & 1u], min(lane & 7, G - 1));
        aca_shuffle<4>(a);
      } else {
        // slots 2 * cta + parity
        ArgMax* mine = part + 2 * (base + g) + (phase & 1u);
        if (tid == 0) *mine = ArgMax{__longlong_as_double(a.v), a.p, __longlong_as_double(a.u)};
        if (!group_barrier(bar + base, G * (phase + 1), Hd->status, abort_flag, Hd->spin)) dead = true;
        // a slot to a thread (every warp reading all of them moved 8 times as much
        // out of L2: 3 us a phase for 589 CTAs), then as above; wb is free again
        // since the barrier
        a = aca_none();
        for (int q = tid; q < G && !dead; q += blockDim.x) {
          const ArgMax* pq = part + 2 * (base + q) + (phase & 1u);
          aca_take(a, AcaBest{__double_as_longlong(__ldcg(&pq->v)), __double_as_longlong(__ldcg(&pq->sv)), __ldcg(&pq->i)});
        }
        aca_shuffle<16>(a);
        if (lane == 0) wb[warp] = a;
        __syncthreads();
        a = wb[lane & 7];
        aca_shuffle<4>(a);
      }
    }
    ++phase;
    return a;
  };
  // acc - sum_{l < k} piv_row[l] (this CTA's entry q of V or U in step l)
  auto residual = [&](double acc, int k, const double* kp, const double* gp) {
    int l = 0;
    if constexpr (KEEP) {
      const int k1 = min(k, kl);
#pragma unroll 4
      for (; l < k1; ++l) acc = __fma_rn(-piv_row[l], kp[l * kstep], acc);
    }
#pragma unroll 4
    for (; l < k; ++l) acc = __fma_rn(-piv_row[l], gp[(size_t)l * n], acc);
    return acc;
  };

  int i = m - 1, k = 0;
  bool hit = false;
  if (m > 0 && p > 0)
    while (true) {
      if (k == cap) { hit = true; break; }
      // residual of row i over this CTA's columns, unnormalised in V[:, k]
      if (tid < k) piv_row[tid] = __ldcg(Bs + (size_t)tid * n + s + i);
      const double xi = x[s + i];
      double first = 0.0;  // (the thread's first entry while the row's U arrives)
      if (c0 + tid < c1) first = kern_entry(kind, kc, xi, x[h + c0 + tid]);
      __syncthreads();
      AcaBest best = aca_none();
      for (int j = c0 + tid; j < c1; j += blockDim.x) {
        const double en = j == c0 + tid ? first : kern_entry(kind, kc, xi, x[h + j]);
        const double acc = residual(en, k, keep + (j - c0), Bs + h + j);
        if (KEEP && k < kl) keep[k * kstep + (j - c0)] = acc;
        else Bs[(size_t)k * n + h + j] = acc;
        // an entry that would win is checked against the used columns (the
        // check runs only then: same result as checking every entry)
        const AcaBest cand{__double_as_longlong(fabs(acc)), 0, 2 * j + (__double2hiint(acc) < 0)};
        if (cand.v > best.v || (cand.v == best.v && cand.p < best.p)) {
          bool used = false;
          for (int l = 0; l < k; ++l) used |= (colp[l] == j);
          if (!used) {
            best.v = cand.v;
            best.p = cand.p;
          }
        }
      }
      best = reduce(best);
      if (dead) return;
      if (best.v <= 0 || best.v > 0x7ff0000000000000LL) break;  // no unused column, a zero row, or not a number
      const int js = best.p >> 1;
      // the pivot column's V entries: V[js, l] (its own CTA's copy in global memory)
      if (tid < k) piv_row[tid] = __ldcg(Bs + (size_t)tid * n + h + js);
      const double rpiv = __ddiv_rn(1.0, aca_value(best));
      const double xj = x[h + js];
      if (r0 + tid < r1) first = kern_entry(kind, kc, x[s + r0 + tid], xj);
      for (int j = c0 + tid; j < c1; j += blockDim.x) {
        double* vp = Bs + (size_t)k * n + h + j;
        if (KEEP && k < kl) *vp = keep[k * kstep + (j - c0)] = __dmul_rn(keep[k * kstep + (j - c0)], rpiv);
        else *vp = __dmul_rn(*vp, rpiv);
      }
      __syncthreads();
      // residual of column js over this CTA's rows, in U[:, k]
      AcaBest nb = aca_none();
      for (int ii = r0 + tid; ii < r1; ii += blockDim.x) {
        const double en = ii == r0 + tid ? first : kern_entry(kind, kc, x[s + ii], xj);
        const double acc = residual(en, k, keep + cc + (ii - r0), Bs + s + ii);
        if (KEEP && k < kl) keep[k * kstep + cc + (ii - r0)] = acc;
        Bs[(size_t)k * n + s + ii] = acc;
        const AcaBest cand{__double_as_longlong(fabs(acc)), 0, 2 * ii + (__double2hiint(acc) < 0)};
        if (cand.v > nb.u) nb.u = cand.v;
        if (cand.v > nb.v || (cand.v == nb.v && cand.p < nb.p)) {
          bool used = (ii == i);
          for (int l = 0; l < k; ++l) used |= (rowp[l] == ii);
          if (!used) {
            nb.v = cand.v;
            nb.p = cand.p;
          }
        }
      }
      nb = reduce(nb);
      if (dead) return;
      if (__longlong_as_double(nb.u) <= eps) break;
      if (tid == 0) {
        rowp[k] = i;
        colp[k] = js;
      }
      __syncthreads();
      ++k;
      if (nb.v < 0) break;
      i = nb.p >> 1;
    }
  if (CL && G > 1) cluster_sync_all();  // no CTA leaves while another may still read its maxima
  if (g == 0 && threadIdx.x == 0) {
    Hd->rank[nid] = k;
    for (int l = 0; l < cap; ++l) {
      Hd->row_piv[nid * cap + l] = l < k ? rowp[l] : -1;
      Hd->col_piv[nid * cap + l] = l < k ? colp[l] : -1;
    }
    if (hit) atomicOr(Hd->status, FIFA_DEV_RANK_CAP);
  }
}

// ---------------------------------------------------------------------------
// ACA of small blocks (both sides <= ACA_WARP_MAX rows): one warp per block,
// eight independent blocks per CTA.  Same arithmetic and pivot rules as k_aca
// (so the same bases, bit for bit); the reductions are warp
// shuffles, with no CTA barrier and no idle warps in them.
// ---------------------------------------------------------------------------
__device__ __forceinline__ ArgMax warp_argmax_all(ArgMax a) {
  for (int o = 16; o > 0; o >>= 1) {
    ArgMax b;
    b.v = __shfl_xor_sync(0xffffffffu, a.v, o);
    b.i = __shfl_xor_sync(0xffffffffu, a.i, o);
    b.sv = __shfl_xor_sync(0xffffffffu, a.sv, o);
    a = am_better(a, b);
  }
  return a;
}

__global__ void __launch_bounds__(256, 3) k_aca_warp(const HmatDesc* __restrict__ Hd, const int4* __restrict__ work,
                                                  int nwork) {
  Hd += blockIdx.y;  // problem of a batched launch (descriptor arrays)
  const int wl = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int item = blockIdx.x * 8 + wl;
  if (item >= nwork) return;  // whole warp
  const int4 w = work[item];
  const int lvl = w.x, bi = w.y;
  const int64_t n = Hd->n;
  const int cap = Hd->cap, kind = Hd->kind;
  const double kc = Hd->kc, eps = Hd->eps;
  const double* __restrict__ x = Hd->x;
  double* Bs = Hd->bases + (size_t)lvl * cap * n;
  int s, h, e;
  node_range(Hd->bnd, lvl, bi, s, h, e);
  const int m = h - s, p = e - h;
  const int nid = node_id(lvl, bi);
  __shared__ int rowp_all[8][FIFA_CAP_MAX], colp_all[8][FIFA_CAP_MAX];
  int* rowp = rowp_all[wl];
  int* colp = colp_all[wl];

  int i = m - 1, k = 0;
  bool hit = false;
  if (m > 0 && p > 0)
    while (true) {
      if (k == cap) { hit = true; break; }
      // residual of row i, stored unnormalised in V[:, k]
      const double xi = x[s + i];
      ArgMax best{-1.0, 0x7fffffff, 0.0};
      for (int j = lane; j < p; j += 32) {
        double acc = kern_entry(kind, kc, xi, x[h + j]);
        for (int l = 0; l < k; ++l)
          acc = __fma_rn(-__ldcg(Bs + (size_t)l * n + s + i), __ldcg(Bs + (size_t)l * n + h + j), acc);
        Bs[(size_t)k * n + h + j] = acc;
        // an entry that would win is checked against the used columns (the
        // check runs only then: same result as checking every entry)
        const ArgMax cand{fabs(acc), j, acc};
        if (am_wins(best, cand)) {
          bool used = false;
          for (int l = 0; l < k; ++l) used |= (colp[l] == j);
          if (!used) best = cand;
        }
      }
      best = warp_argmax_all(best);
      if (!(best.v > 0.0)) break;
      const int js = best.i;
      const double piv = best.sv;
      const double rpiv = __ddiv_rn(1.0, piv);
      for (int j = lane; j < p; j += 32) {
        double* vp = Bs + (size_t)k * n + h + j;
        *vp = __dmul_rn(*vp, rpiv);
      }
      __syncwarp();
      // residual of column js, stored in U[:, k]
      const double xj = x[h + js];
      double umax = 0.0;
      ArgMax nb{-1.0, 0x7fffffff, 0.0};
      for (int ii = lane; ii < m; ii += 32) {
        double acc = kern_entry(kind, kc, x[s + ii], xj);
        for (int l = 0; l < k; ++l)
          acc = __fma_rn(-__ldcg(Bs + (size_t)l * n + s + ii), __ldcg(Bs + (size_t)l * n + h + js), acc);
        Bs[(size_t)k * n + s + ii] = acc;
        umax = nn_max(umax, fabs(acc));
        const ArgMax cand{fabs(acc), ii, acc};
        if (am_wins(nb, cand)) {
          bool used = (ii == i);
          for (int l = 0; l < k; ++l) used |= (rowp[l] == ii);
          if (!used) nb = cand;
        }
      }
      for (int o = 16; o > 0; o >>= 1) umax = nn_max(umax, __shfl_xor_sync(0xffffffffu, umax, o));
      nb = warp_argmax_all(nb);
      if (umax <= eps) break;
      if (lane == 0) {
        rowp[k] = i;
        colp[k] = js;
      }
      __syncwarp();
      ++k;
      if (nb.v < 0.0) break;
      i = nb.i;
    }
  if (lane == 0) {
    Hd->rank[nid] = k;
    for (int l = 0; l < cap; ++l) {
      Hd->row_piv[nid * cap + l] = l < k ? rowp[l] : -1;
      Hd->col_piv[nid * cap + l] = l < k ? colp[l] : -1;
    }
    if (hit) atomicOr(Hd->status, FIFA_DEV_RANK_CAP);
  }
}

// ---------------------------------------------------------------------------
// Host launchers.
// ---------------------------------------------------------------------------
// CTAs of a cluster for each of `blocks` ACA blocks of one launch: up to eight
// while all of them fill the GPU at most four CTAs to an SM, and not more than
// leave 16 rows of a side to a CTA (span: rows and columns of the largest).
static int aca_cluster(int64_t blocks, int span) {
  int c = 1;
  while (c < 8 && 2 * c * blocks <= 608 && span / (4 * c) >= 16) c *= 2;
  return c;
}

// Largest slice of U and V (rows and columns of a CTA) of which steps are kept: with
// fewer than three of them in ACA_KEEP the L1 cache does better.  One assembly, kept /
// not: 312 entries to a CTA 517/566 us, 1000 533/544, 2000 1180/1190, 2500 761/752,
// 3125 1607/1561, 131072 14.85/14.14 ms.
#define ACA_KEEP_SPAN 2048

static cudaError_t launch_aca_cluster(const HmatDesc* Hd, const int4* work, int blocks, int C, int span, cudaStream_t st,
                                      int nprob) {
  const bool keep = span <= ACA_KEEP_SPAN * C;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks * C, nprob);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = keep ? ACA_KEEP * sizeof(double) : 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, keep ? k_aca<true, true> : k_aca<true, false>, Hd, work, C, AcaGroups{},
                            (ArgMax*)nullptr, (unsigned int*)nullptr, (int*)nullptr, (size_t)0);
}

cudaError_t launch_leaf_assemble(const HmatDesc* Hd, int nleaf, cudaStream_t st, int nprob) {
  k_leaf_assemble<<<dim3(nleaf, nprob), 256, 0, st>>>(Hd);
  return cudaGetLastError();
}

// The blocks without a group: work[0, nsolo) the larger ones (span: rows and
// columns of the largest), work[nsolo, nsolo + nwarp) those of at most
// ACA_WARP_MAX rows a side.  Small blocks take one warp each when there are
// enough to fill the GPU, else a cluster each like the larger ones (15 blocks of
// n = 500 took one warp each 278 us), in the same launch if that leaves the
// largest block at most 512 rows and columns to a CTA, two entries of a phase to
// a thread: the two launches of n = 500 took 98 and 87 us one after the other.
cudaError_t launch_aca_blocks(const HmatDesc* Hd, const int4* work, int nsolo, int nwarp, int span, cudaStream_t st,
                              int nprob) {
  const bool small_warps = (int64_t)nwarp * nprob > 608;
  const int together = aca_cluster((int64_t)(nsolo + nwarp) * nprob, span);
  if (!small_warps && nsolo > 0 && nwarp > 0 && span <= 1024 * together)
    return launch_aca_cluster(Hd, work, nsolo + nwarp, together, span, st, nprob);
  if (nsolo > 0) {
    const cudaError_t e = launch_aca_cluster(Hd, work, nsolo, aca_cluster((int64_t)nsolo * nprob, span), span, st, nprob);
    if (e != cudaSuccess) return e;
  }
  if (nwarp <= 0) return cudaSuccess;
  if (!small_warps)
    return launch_aca_cluster(Hd, work + nsolo, nwarp, aca_cluster((int64_t)nwarp * nprob, 2 * ACA_WARP_MAX),
                              2 * ACA_WARP_MAX, st, nprob);
  k_aca_warp<<<dim3((nwarp + 7) / 8, nprob), 256, 0, st>>>(Hd, work + nsolo, nwarp);
  return cudaGetLastError();
}

cudaError_t launch_aca(const HmatDesc* Hd, const int4* work, int ncta, ArgMax* part, unsigned int* bar, int* abort_flag,
                       cudaStream_t st, int nprob, size_t pstride, const AcaGroups* groups) {
  if (ncta <= 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ncta, nprob);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = ACA_KEEP * sizeof(double);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_aca<false, true>, Hd, work, 1, groups ? *groups : AcaGroups{}, part, bar, abort_flag, pstride);
}

int aca_max_coresident_ctas() {
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_aca<false, true>, 256, ACA_KEEP * sizeof(double)) != cudaSuccess)
    per_sm = 1;
  return sms * per_sm;
}

// Device code of the fused applications: leaf steps, the fused sweep and the fused
// H-matrix product, with their launches.  k_apply.cu instantiates the forms that fill
// the GPU, k_apply_cluster.cu those that run as one cluster (two translation units,
// compiled side by side).
#pragma once
#include "fifa_common.cuh"
#include "fifa_launch.h"

#define SW_RHS_MAX 2

template <typename T, int N>
__device__ __forceinline__ T reg_sel(const T (&a)[N], int q) {
  T r = a[0];
#pragma unroll
  for (int t = 1; t < N; ++t)
    if (q == t) r = a[t];
  return r;
}

// ---------------------------------------------------------------------------
// Leaf step of one leaf by one warp, on m entries at vj (global or shared
// memory, element type V), in the factor's precision T (FP64, or FP32 for an
// FP32 copy of a factor: every product and sum in T).  mode 0: v <- L v, 1: v <- L^-1 v, 2: v <- L^T v, 3: v <- L^-T v.
// L column-major (L[i][k] at k*Bm + i, i >= k) with L^T mirrored into the
// upper triangle (L[k][j] at k*Bm + j, j < k): every step reads one contiguous
// column, L's for modes 0 / 1 and L^T's for modes 2 / 3.
// ---------------------------------------------------------------------------
// RPL: rows per lane, 32 RPL >= m; dinv: reciprocal pivots; NR right-hand sides
// (v1 for the second) share the loads of L.  The CH columns after the current
// ones are in flight while those are used: a warp spends 64 cycles on every FP64
// instruction, so a chunk covers the load's latency (64-row leaves: a dependent
// load per column took most of a 30 us substitution).
template <typename T, typename V, int RPL, int CH, int MODE, int NR>
__device__ __forceinline__ void leaf_warp_chunks(const T* __restrict__ Lm, const T* __restrict__ dinv, int Bm, int m,
                                                 V* v0, V* v1, int lane) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr bool subst = MODE == 1 || MODE == 3;
  T x[NR][RPL], o[NR][RPL];
#pragma unroll
  for (int q = 0; q < RPL; ++q) {
    const int i = lane + 32 * q;
    x[0][q] = i < m ? (T)v0[i] : (T)0;
    if (NR > 1) x[NR - 1][q] = i < m ? (T)v1[i] : (T)0;
#pragma unroll
    for (int j = 0; j < NR; ++j) o[j][q] = subst ? x[j][q] : (T)0;
  }
  auto fetch = [&](int t0, T (&c)[CH][RPL], T (&d)[CH]) {
#pragma unroll
    for (int u = 0; u < CH; ++u) {
      const int k = MODE == 3 ? m - 1 - (t0 + u) : t0 + u;
      const bool in = t0 + u < m;
      d[u] = subst && in ? dinv[k] : (T)1;
#pragma unroll
      for (int q = 0; q < RPL; ++q) {
        const int i = lane + 32 * q;
        c[u][q] = in && i < m ? Lm[(size_t)k * Bm + i] : (T)0;
      }
    }
  };
  T cur[CH][RPL], dcur[CH];
  fetch(0, cur, dcur);
  for (int t0 = 0; t0 < m; t0 += CH) {
    T nxt[CH][RPL], dnxt[CH];
    fetch(t0 + CH, nxt, dnxt);
#pragma unroll
    for (int u = 0; u < CH; ++u) {
      if (t0 + u < m) {
        const int k = MODE == 3 ? m - 1 - (t0 + u) : t0 + u;
        T xk[NR];
#pragma unroll
        for (int j = 0; j < NR; ++j) {
          xk[j] = __shfl_sync(FULL, reg_sel<T, RPL>(subst ? o[j] : x[j], k >> 5), k & 31);
          if (subst) xk[j] *= dcur[u];
        }
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
          // whole row groups on the finished side of column k: no arithmetic
          if (MODE == 0 || MODE == 1 ? 32 * q + 31 < k : 32 * q > k) continue;
          const int i = lane + 32 * q;
          const T a = cur[u][q];
#pragma unroll
          for (int j = 0; j < NR; ++j) {
            if (MODE == 0) {
              if (i >= k) o[j][q] += a * xk[j];
            } else if (MODE == 2) {
              if (i <= k) o[j][q] += a * xk[j];
            } else {
              if (i == k) o[j][q] = xk[j];
              else if (MODE == 1 ? i > k : i < k) o[j][q] -= a * xk[j];
            }
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < CH; ++u) {
      dcur[u] = dnxt[u];
#pragma unroll
      for (int q = 0; q < RPL; ++q) cur[u][q] = nxt[u][q];
    }
  }
#pragma unroll
  for (int q = 0; q < RPL; ++q) {
    const int i = lane + 32 * q;
    if (i < m) {
      v0[i] = (V)o[0][q];
      if (NR > 1) v1[i] = (V)o[NR - 1][q];
    }
  }
}

template <typename T, typename V, int RPL, int CH, int NR>
__device__ __forceinline__ void leaf_warp_modes(const T* __restrict__ Lm, const T* __restrict__ dinv, int Bm, int m,
                                                V* v0, V* v1, int mode, int lane) {
  switch (mode) {
    case 0: leaf_warp_chunks<T, V, RPL, CH, 0, NR>(Lm, dinv, Bm, m, v0, v1, lane); break;
    case 1: leaf_warp_chunks<T, V, RPL, CH, 1, NR>(Lm, dinv, Bm, m, v0, v1, lane); break;
    case 2: leaf_warp_chunks<T, V, RPL, CH, 2, NR>(Lm, dinv, Bm, m, v0, v1, lane); break;
    default: leaf_warp_chunks<T, V, RPL, CH, 3, NR>(Lm, dinv, Bm, m, v0, v1, lane); break;
  }
}

// Leaves of at most 32 rows, both right-hand sides at once (v1 nullable).  Lane
// i holds the entries Lm[k Bm + i] of every column k it needs (L[i][k] below
// the diagonal, L[k][i] = L^T mirrored above it), loaded in chunks of CH
// columns before any of them is used, so a chunk's loads are in flight
// together instead of one dependent load per substitution step.  MODE as
// leaf_warp_apply_r.
template <typename T, typename V, int CH, int MODE>
__device__ __forceinline__ void leaf_warp_apply32_m(const T* __restrict__ Lm, const T* __restrict__ dinv, int Bm, int m,
                                                    V* v0, V* v1, int lane) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr bool subst = MODE == 1 || MODE == 3;
  const bool in = lane < Bm;
  const bool two = v1 != nullptr;
  const T x0 = lane < m ? (T)v0[lane] : (T)0;
  const T x1 = (two && lane < m) ? (T)v1[lane] : (T)0;
  const T dl = (subst && in) ? dinv[lane] : (T)1;
  T o0 = subst ? x0 : (T)0, o1 = subst ? x1 : (T)0;
  for (int t0 = 0; t0 < m; t0 += CH) {
    T Lc[CH];
#pragma unroll
    for (int u = 0; u < CH; ++u) {
      const int k = MODE == 3 ? m - 1 - (t0 + u) : t0 + u;
      Lc[u] = (in && t0 + u < m) ? Lm[(size_t)k * Bm + lane] : (T)0;
    }
    const int cnt = min(CH, m - t0);
#pragma unroll
    for (int u = 0; u < CH; ++u) {
      if (u < cnt) {
        const int k = MODE == 3 ? m - 1 - (t0 + u) : t0 + u;
        const T a = Lc[u];
        if (!subst) {  // mode 0: o_i += L[i][k] x_k (i >= k);  mode 2: o_j += L[k][j] x_k (j <= k)
          const T xk0 = __shfl_sync(FULL, x0, k), xk1 = __shfl_sync(FULL, x1, k);
          if (MODE == 0 ? (lane >= k && lane < m) : (lane <= k)) {
            o0 += a * xk0;
            o1 += a * xk1;
          }
        } else {  // mode 1: forward, mode 3: backward substitution with the reciprocal pivots
          const T dk = __shfl_sync(FULL, dl, k);
          const T xk0 = __shfl_sync(FULL, o0, k) * dk, xk1 = __shfl_sync(FULL, o1, k) * dk;
          if (lane == k) {
            o0 = xk0;
            o1 = xk1;
          } else if (MODE == 1 ? (lane > k && lane < m) : (lane < k)) {
            o0 -= a * xk0;
            o1 -= a * xk1;
          }
        }
      }
    }
  }
  if (lane < m) {
    v0[lane] = (V)o0;
    if (two) v1[lane] = (V)o1;
  }
}

template <typename T, typename V>
__device__ __forceinline__ void leaf_warp_apply32(const T* __restrict__ Lm, const T* __restrict__ dinv, int Bm, int m,
                                                  V* v0, V* v1, int mode, int lane) {
  constexpr int CH = sizeof(T) == 4 ? 16 : 8;  // register budget of the fused sweep (64 per thread)
  switch (mode) {
    case 0: leaf_warp_apply32_m<T, V, CH, 0>(Lm, dinv, Bm, m, v0, v1, lane); break;
    case 1: leaf_warp_apply32_m<T, V, CH, 1>(Lm, dinv, Bm, m, v0, v1, lane); break;
    case 2: leaf_warp_apply32_m<T, V, CH, 2>(Lm, dinv, Bm, m, v0, v1, lane); break;
    default: leaf_warp_apply32_m<T, V, CH, 3>(Lm, dinv, Bm, m, v0, v1, lane); break;
  }
}

// Leaves of any size, NR right-hand sides.
template <typename T, typename V, int NR>
__device__ __forceinline__ void leaf_warp_apply(const T* __restrict__ Lm, const T* __restrict__ dinv, int Bm, int m,
                                                V* v0, V* v1, int mode, int lane) {
  if (Bm <= 32) leaf_warp_apply32<T, V>(Lm, dinv, Bm, m, v0, NR > 1 ? v1 : nullptr, mode, lane);
  else if (Bm <= 64) leaf_warp_modes<T, V, 2, 2, NR>(Lm, dinv, Bm, m, v0, v1, mode, lane);
  else  // one at a time: registers
    for (int j = 0; j < NR; ++j)
      leaf_warp_modes<T, V, FIFA_LEAF_MAX / 32, 1, 1>(Lm, dinv, Bm, m, j ? v1 : v0, nullptr, mode, lane);
}

// ---------------------------------------------------------------------------
// Fused sweep: a whole W / W^-1 / W^T / W^-T application in one cooperative
// launch of 2^ls CTAs.  CTA c owns the rows [S, E) of the level-ls node c and
// keeps v on them in shared memory for the whole sweep, so v crosses HBM once
// each way.  The leaves and every level >= ls act inside one CTA (a node there
// lies in one CTA's rows); each level < ls exchanges one partial projection
// per CTA through `part` (its own slots for every level).  Same arithmetic as
// the per-level kernels above:
//   p = [Q_left^T v_left ; Q_right^T v_right],  t = op(Z) p,  v += Q t,
// without its zeros: Z = [0 0; K Y] (the capacitance's factor is [I 0; M^T L2]),
// so t is zero on the left side for Z, and Z^T takes p from the right side
// alone.  A CTA left of the split hands over its partial and goes on; the right
// ones wait for the CTAs of their own node only (a counter per node).  Launched as
// one cluster (contexts with independent CTAs), nothing polls: every CTA passes
// one hardware barrier of the cluster per level.
//
// What bounds it: up to n ~ 2^17 the chain of levels < ls (a barrier of the
// whole grid and loads behind it cost ~17 us per level; now 5 to 8), beyond that
// the FP64 pipe.  So a level's basis rows and its block of Z are copied to
// shared memory while the level before runs (as far as they fit, fs_qcap), and
// sums go over lanes that share an output, not over one thread's chain: a lone
// warp takes 64 cycles per FP64 instruction.  One W^-1 of n = 2^20 to two
// vectors 1.06 -> 0.83 ms; a solve of n = 500 129 -> 61 us.
// ---------------------------------------------------------------------------
#define FS_WARPS 8
// Entries of a level's basis rows staged ahead, by the CTA's rows: as many as
// leave four CTAs to an SM up to 160 rows, two up to 512; CTAs of more rows
// stage nothing (their levels are long).
__host__ __device__ inline int fs_qcap(int rows) { return rows <= 160 ? 1536 : (rows <= 512 ? 4608 : 0); }
#define FS_ZBUF 512         // doubles of a level's Z block staged ahead: 2 r^2, r <= 16

// Ask L2 to fetch the 128-byte line holding p (no data is returned; p must
// point into an allocation).
__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// Prefetch the basis columns a < r of level l on rows [a0, a1) into L2, the
// CTA's threads sharing the lines.
template <typename T>
__device__ __forceinline__ void prefetch_cols_l2(const T* __restrict__ Qb, int64_t n, int r, int a0, int a1) {
  constexpr int PER = 128 / (int)sizeof(T);
  const int first = a0 / PER, last = (a1 - 1) / PER;
  if (a1 <= a0) return;
  const int nl = last - first + 1;
  for (int t = threadIdx.x; t < r * nl; t += blockDim.x) {
    const int a = t / nl, li = first + t % nl;
    prefetch_l2(Qb + (size_t)a * n + (size_t)li * PER);
  }
}

// Sum over rows [a0, a1) of Bl[col][p] * xs[j][p - S] for K outputs
// o = (unit, c, j) described by fn(o, &a0, &a1, &col, &j) (col < 0: skip);
// results to out[o], accumulated in TX.  Threads take (output, row chunk)
// pairs; chunk partials are combined in a fixed order.
template <typename TB, typename TX, typename F>
__device__ void tile_dots(int K, const TB* __restrict__ Bl, int64_t n, const TX* xs, int rows, int S, F fn,
                          TX* red, TX* out) {
  const int nt = blockDim.x;
  const int nch = K >= nt ? 1 : nt / K;
  for (int o0 = 0; o0 < K; o0 += nt) {
    const int kk = min(nt, K - o0);
    const int ch = nch == 1 ? 0 : threadIdx.x / kk;
    const int o = o0 + (nch == 1 ? threadIdx.x : threadIdx.x % kk);
    TX acc = (TX)0;
    if ((nch == 1 && threadIdx.x < kk) || (nch > 1 && ch < nch)) {
      int a0, a1, col, j;
      fn(o, a0, a1, col, j);
      if (col >= 0) {
        const TB* b = Bl + (size_t)col * n;
        const TX* xj = xs + (size_t)j * rows - S;
#pragma unroll 8
        for (int p = a0 + ch; p < a1; p += nch) acc += (TX)b[p] * xj[p];
      }
    }
    __syncthreads();
    if (nch > 1) {
      if (ch < nch) red[ch * kk + (threadIdx.x % kk)] = acc;
      __syncthreads();
      if ((int)threadIdx.x < kk) {
        TX v = (TX)0;
        for (int q = 0; q < nch; ++q) v += red[q * kk + threadIdx.x];
        out[o0 + threadIdx.x] = v;
      }
    } else if ((int)threadIdx.x < kk) {
      out[o] = acc;
    }
    __syncthreads();
  }
}

#define FS_BUF 512  // entries of node projections (and of op(Z) p) per batch

// Shared scratch carved after v; T is the arithmetic type of the sweep.
template <typename T>
struct FsShared {
  T* pj;                  // FS_BUF: projections p of a batch of nodes
  T* tv;                  // FS_BUF: t = op(Z) p of the batch
  T* red;                 // 256 reduction partials
  double* zb;             // 2 x FS_ZBUF: staged blocks of Z
  T* qb;                  // 2 x qcap: staged basis rows
  int qcap;               // (0: none)
  unsigned short* lmap;   // rows: local leaf of each row
};

// basis columns whose loads a thread issues together (fewer FP64 ones: the
// register budget of the fused sweep is 64 per thread)
#define FS_RG_OF(T) (sizeof(T) == 4 ? 4 : 2)

// v_p += sum_{a < r} Q[a][p] t[a] for one row p (two right-hand sides in acc0,
// acc1; t interleaved by right-hand side), FS_RG_OF(T) loads in flight at a time.
template <typename T, int NR>
__device__ __forceinline__ void fs_row_update(const T* __restrict__ Qb, int64_t n, int p, int r, const T* tn, T& acc0,
                                              T& acc1) {
  constexpr int nrhs = NR;
  constexpr int RG = FS_RG_OF(T);
  for (int a0 = 0; a0 < r; a0 += RG) {
    T q[RG];
#pragma unroll
    for (int u = 0; u < RG; ++u) q[u] = a0 + u < r ? Qb[(size_t)(a0 + u) * n + p] : (T)0;
#pragma unroll
    for (int u = 0; u < RG; ++u) {
      if (a0 + u < r) {
        acc0 += q[u] * tn[(a0 + u) * nrhs];
        if (nrhs > 1) acc1 += q[u] * tn[(a0 + u) * nrhs + 1];
      }
    }
  }
}

// One level >= ls inside CTA c (rows [S, S + R)): the level's nodes in c's
// subtree in batches whose projections fit FS_BUF; each batch takes one pass of
// dot products (output-major, no cross-lane reductions), t = op(Z) p per
// node, and the row update v += Q t.  All arithmetic in T.
template <typename T, int NR>
__device__ void fs_local_level(const FactDesc* __restrict__ Fd, int l, int ls, int c, T* vs, int rows, int S,
                               int R, int zsel, int zt, FsShared<T>& sh) {
  constexpr int nrhs = NR;
  const int L = Fd->L, cap = Fd->cap, ld2 = 2 * cap;
  const int64_t n = Fd->n;
  const int* bnd = Fd->bnd;
  const int nsub = 1 << (l - ls), i0 = c << (l - ls);
  const T* Qb = (const T*)Fd->Q + (size_t)l * cap * n;
  int rmax = 0;
  for (int q = 0; q < nsub; ++q) rmax = max(rmax, Fd->rank[node_id(l, i0 + q)]);
  if (rmax == 0) return;
  // Z: p of both sides, t of the right one; Z^T: p of the right side, t of both
  const int half = rmax * nrhs, np = zt ? half : 2 * half, ntt = zt ? 2 * half : half;  // entries per node
  const int nb = max(1, FS_BUF / (2 * half));
  for (int b0 = 0; b0 < nsub; b0 += nb) {
    const int bn = min(nb, nsub - b0);
    tile_dots<T, T>(bn * np, Qb, n, vs, rows, S,
                    [&](int o, int& a0, int& a1, int& col, int& j) {
                      const int node = o / np, rem = o % np, side = zt ? 1 : rem / half, aj = rem % half;
                      const int a = aj / nrhs;
                      j = aj % nrhs;
                      int s0, h0, e0;
                      node_range(bnd, l, i0 + b0 + node, s0, h0, e0);
                      a0 = side ? h0 : s0;
                      a1 = side ? e0 : h0;
                      col = a < Fd->rank[node_id(l, i0 + b0 + node)] ? a : -1;
                    },
                    sh.red, sh.pj);
    for (int k = threadIdx.x; k < bn * ntt; k += blockDim.x) {
      const int node = k / ntt, rem = k % ntt, j = rem % nrhs;
      const int side = zt ? rem / half : 1, a = (rem % half) / nrhs;
      const int nid = node_id(l, i0 + b0 + node);
      const int r = Fd->rank[nid];
      T acc = (T)0;
      if (a < r) {
        const double* Z = (zsel ? Fd->Zi : Fd->Zf) + (size_t)nid * ld2 * ld2;
        const T* pn = sh.pj + node * np;
        if (zt) {
          for (int b = 0; b < r; ++b) acc += (T)Z[(r + b) * ld2 + side * r + a] * pn[b * nrhs + j];
        } else {
          for (int b = 0; b < r; ++b) acc += (T)Z[(r + a) * ld2 + b] * pn[b * nrhs + j];
          for (int b = 0; b < r; ++b) acc += (T)Z[(r + a) * ld2 + r + b] * pn[half + b * nrhs + j];
        }
      }
      sh.tv[k] = acc;
    }
    __syncthreads();
    for (int p = S + (int)threadIdx.x; p < S + R; p += blockDim.x) {
      const int node = ((int)sh.lmap[p - S] >> (L - l)) - b0;
      if (node < 0 || node >= bn) continue;
      const int gi = i0 + b0 + node;
      const int r = Fd->rank[node_id(l, gi)];
      int s0, h0, e0;
      node_range(bnd, l, gi, s0, h0, e0);
      if (!zt && p < h0) continue;
      const T* tn = sh.tv + node * ntt + (zt && p >= h0 ? half : 0);
      // the products accumulate onto v itself (no separate add per row)
      T acc0 = vs[p - S], acc1 = nrhs > 1 ? vs[rows + p - S] : (T)0;
      fs_row_update<T, NR>(Qb, n, p, r, tn, acc0, acc1);
      vs[p - S] = acc0;
      if (nrhs > 1) vs[rows + p - S] = acc1;
    }
    __syncthreads();
  }
}

// Asynchronous copies into shared memory.
__device__ __forceinline__ void fs_copy(double* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void fs_copy(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Start copying what level l < ls needs besides v into buffer b: the CTA's rows
// of its r basis columns and rows r .. 2r of the node's Z (one group of copies,
// empty if they do not fit).
template <typename T>
__device__ void fs_stage(const FactDesc* __restrict__ Fd, int l, int ls, int c, int r, int S, int R, int zsel, int b,
                         FsShared<T>& sh) {
  if (r * R <= sh.qcap && 2 * r * r <= FS_ZBUF) {
    const int cap = Fd->cap, ld2 = 2 * cap;
    const int64_t n = Fd->n;
    const T* Qb = (const T*)Fd->Q + (size_t)l * cap * n + S;
    const double* Z = (zsel ? Fd->Zi : Fd->Zf) + (size_t)node_id(l, c >> (ls - l)) * ld2 * ld2;
    for (int t = threadIdx.x; t < r * R; t += blockDim.x) {
      const int a = t / R, p = t - a * R;
      fs_copy(sh.qb + b * sh.qcap + t, Qb + (size_t)a * n + p);
    }
    for (int t = threadIdx.x; t < 2 * r * r; t += blockDim.x) {
      const int a = t / (2 * r), q = t - a * 2 * r;
      fs_copy(sh.zb + b * FS_ZBUF + t, Z + (size_t)(r + a) * ld2 + q);
    }
  } else if (sizeof(T) == 4) {  // FP32 levels are memory-bound: into L2 at least
    prefetch_cols_l2<T>((const T*)Fd->Q + (size_t)l * Fd->cap * Fd->n, Fd->n, r, S, S + R);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// Sum over a power of two of neighbouring lanes; every one of them gets it.
template <typename T>
__device__ __forceinline__ T lanes_sum(T v, int width) {
  for (int o = width >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Lanes per output when K outputs share 256 threads: a power of two, 1 .. 32.
__device__ __forceinline__ int lanes_for(int K) {
  int w = 32;
  while (w > 1 && w * K > 256) w >>= 1;
  return w;
}

// One level < ls: node i = c >> (ls - l) spans 2^(ls - l) CTAs; c's rows lie in
// one child (side).  The CTAs hand over their partial projections in FP64
// (`part`, this level's slots) and count themselves in at their node's counter.
// What the level needs is in buffer `buf` (fs_stage, the oldest group of
// copies) or still in global memory.  CL: the launch's CTAs are one cluster and
// meet at its barrier instead, all of them at every level.  Returns false if the
// wait gave up.
template <typename T, int NR, bool CL>
__device__ bool fs_global_level(const FactDesc* __restrict__ Fd, int l, int ls, int c, int r, T* vs, int rows, int S,
                                int E, int zsel, int zt, double* __restrict__ part, int buf, unsigned int* counter,
                                int* abort_flag, FsShared<T>& sh) {
  constexpr int nrhs = NR;
  const int tid = threadIdx.x, R = E - S;
  const int cap = Fd->cap, ld2 = 2 * cap, pstr = cap * SW_RHS_MAX;
  const int64_t n = Fd->n;
  const int span = ls - l, i = c >> span, side = (c >> (span - 1)) & 1, half = 1 << (span - 1), c0 = i << span;
  const int nid = node_id(l, i);
  const bool staged = r * R <= sh.qcap && 2 * r * r <= FS_ZBUF;
  asm volatile("cp.async.wait_group 1;" ::: "memory");  // this level's copies; the next level's may be in flight
  __syncthreads();                                       // ... every thread's, and v is up to date
  if (r == 0) {                                          // (for every CTA of the node: none waits)
    if constexpr (CL) cluster_sync_all();                // (other nodes of the level may have a rank)
    return true;
  }
  const T* Qb = (const T*)Fd->Q + (size_t)l * cap * n;
  const T* q = staged ? sh.qb + buf * sh.qcap : Qb + S;  // column a at q + a * qs, from row S
  const size_t qs = staged ? (size_t)R : (size_t)n;
  const double* Z = staged ? sh.zb + buf * FS_ZBUF
                           : (zsel ? Fd->Zi : Fd->Zf) + (size_t)nid * ld2 * ld2 + (size_t)r * ld2;
  const int zs = staged ? 2 * r : ld2;  // row a of Z's lower half at Z + a * zs
  const int K = r * nrhs;
  if (!zt || side) {
    // this CTA's partial p: neighbouring lanes share a column, rows striding
    const int w = lanes_for(r), ch = tid & (w - 1);
    for (int o0 = 0; o0 < r; o0 += 256 / w) {
      const int a = o0 + tid / w;
      T acc0 = (T)0, acc1 = (T)0;
      if (a < r) {
        const T* qa = q + (size_t)a * qs;
        constexpr int IN_FLIGHT = sizeof(T) == 4 ? 16 : 8;
#pragma unroll IN_FLIGHT
        for (int p = ch; p < R; p += w) {
          const T qv = qa[p];
          acc0 += qv * vs[p];
          if (nrhs > 1) acc1 += qv * vs[rows + p];
        }
      }
      acc0 = lanes_sum(acc0, w);
      if (nrhs > 1) acc1 = lanes_sum(acc1, w);
      if (ch == 0 && a < r) {
        __stcg(part + (size_t)c * pstr + a * nrhs, (double)acc0);
        if (nrhs > 1) __stcg(part + (size_t)c * pstr + a * nrhs + 1, (double)acc1);
      }
    }
    __syncthreads();
    if (!CL && tid == 0) {
      __threadfence();
      atomicAdd(counter, 1u);
    }
  }
  if constexpr (CL) cluster_sync_all();
  if (!zt && !side) return true;  // the left rows keep their values
  // wait for the CTAs that hand over: both halves, or the right one
  __shared__ int arrived;
  if (!CL && tid == 0) {
    const unsigned int target = zt ? half : 2 * half;
    const unsigned int limit = Fd->spin ? Fd->spin : FIFA_SPIN_LIMIT;
    unsigned int spins = 0;
    int ok = 1;
    while (*((volatile unsigned int*)counter) < target) {
      if (*((volatile int*)abort_flag)) {
        ok = 0;
        break;
      }
      if (++spins > limit) {
        atomicOr(Fd->status, FIFA_DEV_TIMEOUT);
        *((volatile int*)abort_flag) = 1;
        ok = 0;
        break;
      }
      if (spins > 256) __nanosleep(64);
    }
    __threadfence();
    arrived = ok;
  }
  if constexpr (!CL) {
    __syncthreads();
    if (!arrived) return false;
  }
  // p (left entries, then right ones; right ones alone for Z^T)
  {
    const int K2 = zt ? K : 2 * K, w = lanes_for(K2), ch = tid & (w - 1);
    for (int o0 = 0; o0 < K2; o0 += 256 / w) {
      const int o = o0 + tid / w;
      double acc = 0.0;
      if (o < K2) {
        const int sd = zt ? 1 : o / K, k = o - (zt ? 0 : sd * K);
        const double* src = part + (size_t)(c0 + sd * half) * pstr + k;
#pragma unroll 4
        for (int g = ch; g < half; g += w) acc += __ldcg(src + (size_t)g * pstr);
      }
      acc = lanes_sum(acc, w);
      if (ch == 0 && o < K2) sh.pj[o] = (T)acc;
    }
  }
  __syncthreads();
  // t on this CTA's side
  {
    const int w = lanes_for(K), ch = tid & (w - 1), terms = zt ? r : 2 * r;
    for (int o0 = 0; o0 < K; o0 += 256 / w) {
      const int o = o0 + tid / w, a = o / nrhs, j = o % nrhs;
      T acc = (T)0;
      if (o < K)
        for (int b = ch; b < terms; b += w)
          acc += (T)(zt ? Z[b * zs + side * r + a] : Z[a * zs + b]) * sh.pj[b * nrhs + j];
      acc = lanes_sum(acc, w);
      if (ch == 0 && o < K) sh.tv[o] = acc;
    }
  }
  __syncthreads();
  if (staged) {
    for (int t = tid; t < R * nrhs; t += blockDim.x) {
      const int j = t >= R ? 1 : 0, p = t - j * R;
      T acc = vs[(size_t)j * rows + p];
      for (int a = 0; a < r; ++a) acc += q[a * R + p] * sh.tv[a * nrhs + j];
      vs[(size_t)j * rows + p] = acc;
    }
  } else {
#pragma unroll 2
    for (int p = S + tid; p < E; p += blockDim.x) {
      T acc0 = vs[p - S], acc1 = nrhs > 1 ? vs[rows + p - S] : (T)0;
      fs_row_update<T, NR>(Qb, n, p, r, sh.tv, acc0, acc1);
      vs[p - S] = acc0;
      if (nrhs > 1) vs[rows + p - S] = acc1;
    }
  }
  return true;
}

template <typename T, int NR>
__device__ void fs_leaves(const FactDesc* __restrict__ Fd, int ls, int c, T* vs, int rows, int S, int mode) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int L = Fd->L, Bm = Fd->Bm;
  const int nl = 1 << (L - ls), first = c << (L - ls);
  for (int q = warp; q < nl; q += FS_WARPS) {
    const int leaf = first + q;
    const int s = Fd->bnd[bnd_off(L) + leaf], e = Fd->bnd[bnd_off(L) + leaf + 1];
    const T* Lm = (const T*)Fd->Lleaf + (size_t)leaf * Bm * Bm;
    const T* dinv = (const T*)Fd->Ldinv + (size_t)leaf * Bm;
    leaf_warp_apply<T, T, NR>(Lm, dinv, Bm, e - s, vs + (s - S), vs + rows + (s - S), mode, lane);
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// Warp-owned subtrees.  Below the fused level ls every warp of the CTA owns
// the subtree of one level-lw node, lw = min(L, ls + FS_WL) (eight warps: three
// levels), and applies the leaves and the levels >= lw of that subtree alone:
// lanes stride over the node's rows, projections are reduced with warp
// shuffles, and no block barrier is passed.  Levels ls <= l < lw combine one
// partial projection per warp through shared memory with one block barrier
// per level.  The per-warp arrays: p and t of the current node (pj, 2 FS_WSL
// entries per warp) and the warp partials of the block levels (tv, two
// buffers alternating by level).  Ranks above FS_RFAST(T, NR) take the
// block-wide path instead.  FP32 only: in FP64 the shuffle reductions (two
// 32-bit shuffles and a DADD per step) cost more FP64 issue than the block
// barriers they replace (the FP64 W^-1 sweep at n = 2^20: 1.06 ms block-wide,
// 1.21 ms warp-owned).
// ---------------------------------------------------------------------------
#define FS_WARP_OWNED(T, NR) (sizeof(T) == 4)
#define FS_WL 3
#define FS_WSL 32                                           // p or t entries per warp: 2 r nrhs <= 32
#define FS_RFAST(T, NR) ((sizeof(T) == 4 ? 16 : 8) / (NR))  // ranks the warp path takes

template <typename T>
__device__ __forceinline__ T warp_allsum(T v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// t = op(Z) p for a node of rank r: lane k < 2 r nrhs computes t[k]
// (k = (row, j)); p and t interleaved by right-hand side.  Z's upper half is
// zero: t of the right side alone for Z, p of the right side alone for Z^T.
template <typename T, int NR>
__device__ __forceinline__ void fw_apply_z(const double* __restrict__ Z, int ld2, int r, int zt, const T* pw, T* tw,
                                           int lane) {
  constexpr int nrhs = NR;
  if (lane < 2 * r * nrhs && (zt || lane >= r * nrhs)) {
    const int row = lane / nrhs, j = lane % nrhs;
    T acc = (T)0;
    for (int b = zt ? r : 0; b < 2 * r; ++b) acc += (T)(zt ? Z[b * ld2 + row] : Z[row * ld2 + b]) * pw[b * nrhs + j];
    tw[lane] = acc;
  }
  __syncwarp();
}

// Projection of rows [a0, a1) onto the r columns of Qb, accumulated per lane
// (rows lane, lane + 32, ...) and reduced over the warp; every lane ends with
// the sums, lane 0 stores them at out[a nrhs + j].
template <typename T, int NR>
__device__ __forceinline__ void fw_project(const T* __restrict__ Qb, int64_t n, int r, const T* vs, int rows, int S,
                                           int a0, int a1, T* out, int lane) {
  constexpr int nrhs = NR;
  constexpr int CG = 8 / NR;  // columns per pass over the rows (registers: CG NR accumulators)
  for (int c0 = 0; c0 < r; c0 += CG) {
    T acc[CG][NR];
#pragma unroll
    for (int a = 0; a < CG; ++a)
#pragma unroll
      for (int j = 0; j < NR; ++j) acc[a][j] = (T)0;
    for (int p = a0 + lane; p < a1; p += 32) {
      T v[NR];
#pragma unroll
      for (int j = 0; j < NR; ++j) v[j] = vs[(size_t)j * rows + p - S];
      T q[CG];
#pragma unroll
      for (int a = 0; a < CG; ++a) q[a] = c0 + a < r ? Qb[(size_t)(c0 + a) * n + p] : (T)0;
#pragma unroll
      for (int a = 0; a < CG; ++a)
        if (c0 + a < r)
#pragma unroll
          for (int j = 0; j < NR; ++j) acc[a][j] += q[a] * v[j];
    }
#pragma unroll
    for (int a = 0; a < CG; ++a)
      if (c0 + a < r)
#pragma unroll
        for (int j = 0; j < NR; ++j) {
          const T t = warp_allsum(acc[a][j]);
          if (lane == 0) out[(c0 + a) * nrhs + j] = t;
        }
  }
}

// v_p += sum_a Q[a][p] t[(off + a) nrhs + j] for rows [a0, a1), lanes striding.
template <typename T, int NR>
__device__ __forceinline__ void fw_update(const T* __restrict__ Qb, int64_t n, int r, T* vs, int rows, int S, int a0,
                                          int a1, const T* tw, int off) {
  const int lane = threadIdx.x & 31;
#pragma unroll 2
  for (int p = a0 + lane; p < a1; p += 32) {
    T acc0 = vs[p - S], acc1 = NR > 1 ? vs[rows + p - S] : (T)0;
    fs_row_update<T, NR>(Qb, n, p, r, tw + off * NR, acc0, acc1);
    vs[p - S] = acc0;
    if (NR > 1) vs[rows + p - S] = acc1;
  }
}

// One node of a warp-owned level: projection of both sides, t = op(Z) p, update.
template <typename T, int NR>
__device__ void fw_node(const FactDesc* __restrict__ Fd, int l, int i, T* vs, int rows, int S, int zsel, int zt,
                        T* pw, T* tw, int lane) {
  const int cap = Fd->cap, ld2 = 2 * cap;
  const int64_t n = Fd->n;
  const int nid = node_id(l, i);
  const int r = Fd->rank[nid];
  if (r == 0) return;
  int s0, h0, e0;
  node_range(Fd->bnd, l, i, s0, h0, e0);
  const T* Qb = (const T*)Fd->Q + (size_t)l * cap * n;
  if (!zt) fw_project<T, NR>(Qb, n, r, vs, rows, S, s0, h0, pw, lane);
  fw_project<T, NR>(Qb, n, r, vs, rows, S, h0, e0, pw + r * NR, lane);
  __syncwarp();
  fw_apply_z<T, NR>((zsel ? Fd->Zi : Fd->Zf) + (size_t)nid * ld2 * ld2, ld2, r, zt, pw, tw, lane);
  if (zt) fw_update<T, NR>(Qb, n, r, vs, rows, S, s0, h0, tw, 0);
  fw_update<T, NR>(Qb, n, r, vs, rows, S, h0, e0, tw, r);
  __syncwarp();
}

// The leaves and levels >= lw of warp w's subtree (root node wi at level lw),
// in the sweep's order: up = leaves first, then levels L-1 .. lw; else the
// levels lw .. L-1, then the leaves.
template <typename T, int NR>
__device__ void fw_subtree(const FactDesc* __restrict__ Fd, int lw, int wi, T* vs, int rows, int S, int mode, bool up,
                           int zsel, int zt, T* pw, T* tw, int lane) {
  const int L = Fd->L, Bm = Fd->Bm;
  auto leaves = [&]() {
    const int nl = 1 << (L - lw), first = wi << (L - lw);
    for (int q = 0; q < nl; ++q) {
      const int leaf = first + q;
      const int s = Fd->bnd[bnd_off(L) + leaf], e = Fd->bnd[bnd_off(L) + leaf + 1];
      const T* Lm = (const T*)Fd->Lleaf + (size_t)leaf * Bm * Bm;
      const T* dinv = (const T*)Fd->Ldinv + (size_t)leaf * Bm;
      leaf_warp_apply<T, T, NR>(Lm, dinv, Bm, e - s, vs + (s - S), vs + rows + (s - S), mode, lane);
      __syncwarp();
    }
  };
  if (up) {
    leaves();
    for (int l = L - 1; l >= lw; --l)
      for (int q = 0; q < (1 << (l - lw)); ++q) fw_node<T, NR>(Fd, l, (wi << (l - lw)) + q, vs, rows, S, zsel, zt, pw, tw, lane);
  } else {
    for (int l = lw; l < L; ++l)
      for (int q = 0; q < (1 << (l - lw)); ++q) fw_node<T, NR>(Fd, l, (wi << (l - lw)) + q, vs, rows, S, zsel, zt, pw, tw, lane);
    leaves();
  }
}

// One level ls <= l < lw: warp w's rows (those of its level-lw node) lie in
// one side of a level-l node; one partial per warp in shared memory, one block
// barrier, then every warp forms p from its node's warps (fixed order),
// t = op(Z) p and updates its own rows.  nsub: warps that own a subtree.
template <typename T, int NR>
__device__ void fw_block_level(const FactDesc* __restrict__ Fd, int l, int lw, int c, int nsub, T* vs, int rows,
                               int S, int zsel, int zt, T* part, T* pw, T* tw, int warp, int lane) {
  constexpr int nrhs = NR;
  const int cap = Fd->cap, ld2 = 2 * cap;
  const int64_t n = Fd->n;
  const bool own = warp < nsub;
  const int wi = (c * nsub) + warp;           // the warp's level-lw node
  const int span = lw - l, i = wi >> span;    // its level-l node
  const int nid = node_id(l, i);
  const int r = Fd->rank[nid];
  const T* Qb = (const T*)Fd->Q + (size_t)l * cap * n;
  const int side = (wi >> (span - 1)) & 1;
  if (own && r > 0 && (!zt || side)) {
    const int a0 = Fd->bnd[bnd_off(lw) + wi], a1 = Fd->bnd[bnd_off(lw) + wi + 1];
    fw_project<T, NR>(Qb, n, r, vs, rows, S, a0, a1, part + warp * FS_WSL, lane);
  }
  __syncthreads();
  if (!own || r == 0 || (!zt && !side)) return;
  // warps of node i: [i << span, (i + 1) << span) - c nsub, left half first
  const int w0 = (i << span) - c * nsub, half = 1 << (span - 1);
  if (lane < 2 * r * nrhs && (!zt || lane >= r * nrhs)) {
    const int sd = lane / (r * nrhs), k = lane % (r * nrhs);
    T acc = (T)0;
    for (int q = 0; q < half; ++q) acc += part[(w0 + sd * half + q) * FS_WSL + k];
    pw[lane] = acc;
  }
  __syncwarp();
  fw_apply_z<T, NR>((zsel ? Fd->Zi : Fd->Zf) + (size_t)nid * ld2 * ld2, ld2, r, zt, pw, tw, lane);
  const int a0 = Fd->bnd[bnd_off(lw) + wi], a1 = Fd->bnd[bnd_off(lw) + wi + 1];
  fw_update<T, NR>(Qb, n, r, vs, rows, S, a0, a1, tw, side * r);
  __syncwarp();
}

// mode 0: v <- W v, 1: W^-1 v, 2: W^T v, 3: W^-T v; mode 4: v <- W^-T W^-1 v
// (both inverse sweeps, v kept in shared memory in between: a full solve with
// the factor).  Arithmetic in T: FP64 for an FP64 factor, FP32 for an FP32
// copy (the global v stays FP64, converted on load and store).  active
// (nullable): when *active == 0 the launch does nothing (a converged
// iteration).  Dynamic shared memory: nrhs * rows entries of T (rows >= the
// longest level-ls node), then the FsShared arrays.  vlist (nullable): several
// factors of one plan in one launch, problem blockIdx.y: its descriptor
// Fd[blockIdx.y], its vector vlist[blockIdx.y], its partials, barrier and
// abort flag pstride bytes after the previous problem's.  CL: the grid is one
// cluster (bar and abort_flag are not used then; an instantiation of its own, since
// a switch at run time cost the other forms 1%: a draw of n = 65537 968 -> 978 us).
template <typename T, int NR, bool BATCH = false, bool CL = false>
__global__ void __launch_bounds__(256, 4) k_sweep_fused(const FactDesc* __restrict__ Fd, double* __restrict__ v,
                                                        int mode, int ls, int rows, double* __restrict__ part,
                                                        unsigned int* __restrict__ bar, int* __restrict__ abort_flag,
                                                        const int* __restrict__ active, double* const* vlist,
                                                        size_t pstride) {
  constexpr int nrhs = NR;
  if (active && *active == 0) return;
  // (a separate instantiation: re-pointed arguments live in registers for the
  // whole kernel, which the single-problem kernels cannot afford)
  if constexpr (BATCH) {
    Fd += blockIdx.y;
    v = vlist[blockIdx.y];
    part = (double*)((char*)part + blockIdx.y * pstride);
    bar = (unsigned int*)((char*)bar + blockIdx.y * pstride);
    abort_flag = (int*)((char*)abort_flag + blockIdx.y * pstride);
  }
  extern __shared__ __align__(16) unsigned char fs_smem[];
  T* vs = (T*)fs_smem;
  FsShared<T> sh;
  sh.pj = vs + (size_t)rows * nrhs;
  sh.tv = sh.pj + FS_BUF;
  sh.red = sh.tv + FS_BUF;
  sh.zb = (double*)(((uintptr_t)(sh.red + 256) + 7) & ~(uintptr_t)7);
  sh.qcap = fs_qcap(rows);
  sh.qb = (T*)(sh.zb + (sh.qcap ? 2 * FS_ZBUF : 0));
  sh.lmap = (unsigned short*)(sh.qb + 2 * sh.qcap);
  const int c = blockIdx.x;
  const int L = Fd->L;
  const int64_t n = Fd->n;
  const int S = Fd->bnd[bnd_off(ls) + c], E = Fd->bnd[bnd_off(ls) + c + 1];
  // warp-owned subtrees when every rank of the CTA's levels >= ls is small
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int lw = min(L, ls + FS_WL), nsub = 1 << (lw - ls);
  __shared__ int rk_big;
  __shared__ int rkg[FIFA_LEVELS_MAX];  // this CTA's node's rank at each level < ls
  if (threadIdx.x == 0) rk_big = 0;
  if ((int)threadIdx.x < ls) rkg[threadIdx.x] = Fd->rank[node_id(threadIdx.x, c >> (ls - threadIdx.x))];
  for (int j = 0; j < nrhs; ++j)
    for (int p = threadIdx.x; p < E - S; p += blockDim.x) vs[(size_t)j * rows + p] = (T)v[(size_t)j * n + S + p];
  __syncthreads();
  __shared__ int rml[FIFA_LEVELS_MAX];  // the largest rank of each local level in this CTA
  if constexpr (FS_WARP_OWNED(T, NR)) {
    for (int l = threadIdx.x; l < FIFA_LEVELS_MAX; l += blockDim.x) rml[l] = 0;
    __syncthreads();
    for (int l = ls; l < L; ++l)
      for (int q = threadIdx.x; q < (1 << (l - ls)); q += blockDim.x) {
        const int rq = Fd->rank[node_id(l, (c << (l - ls)) + q)];
        if (rq > FS_RFAST(T, NR)) rk_big = 1;
        atomicMax(&rml[l], rq);
      }
  }
  __syncthreads();
  // FP32: the CTA's basis rows of every local level, fetched into L2 ahead of
  // use (measured: 4% off the preconditioner solve; in FP64 the prefetches
  // cost more than they save)
  if constexpr (FS_WARP_OWNED(T, NR))
    for (int l = ls; l < L; ++l) prefetch_cols_l2<T>((const T*)Fd->Q + (size_t)l * Fd->cap * n, n, rml[l], S, E);
  const bool fast = FS_WARP_OWNED(T, NR) && !rk_big && nsub <= FS_WARPS;
  if (!fast) {  // the block-wide path: the local leaf of every row
    const int nl = 1 << (L - ls), first = c << (L - ls);
    for (int q = threadIdx.x; q < nl; q += blockDim.x) {
      const int s0 = Fd->bnd[bnd_off(L) + first + q], e0 = Fd->bnd[bnd_off(L) + first + q + 1];
      for (int p = s0; p < e0; ++p) sh.lmap[p - S] = (unsigned short)q;
    }
    __syncthreads();
  }
  bool ok = true;
  T* pw = sh.pj + warp * 2 * FS_WSL;  // p of the warp's node
  T* tw = pw + FS_WSL;                // t of the warp's node
  auto local_up = [&](int md, int zsel, int zt) {
    if (!fast) {
      fs_leaves<T, NR>(Fd, ls, c, vs, rows, S, md);
      for (int l = L - 1; l >= ls; --l) fs_local_level<T, NR>(Fd, l, ls, c, vs, rows, S, E - S, zsel, zt, sh);
      return;
    }
    if constexpr (FS_WARP_OWNED(T, NR)) {
      if (warp < nsub)
        fw_subtree<T, NR>(Fd, lw, (c << (lw - ls)) + warp, vs, rows, S, md, true, zsel, zt, pw, tw, lane);
      for (int l = lw - 1; l >= ls; --l)
        fw_block_level<T, NR>(Fd, l, lw, c, nsub, vs, rows, S, zsel, zt, sh.tv + (l & 1) * FS_WARPS * FS_WSL, pw, tw,
                              warp, lane);
      __syncthreads();
    }
  };
  auto local_down = [&](int md, int zsel, int zt) {
    if (!fast) {
      for (int l = ls; l < L; ++l) fs_local_level<T, NR>(Fd, l, ls, c, vs, rows, S, E - S, zsel, zt, sh);
      fs_leaves<T, NR>(Fd, ls, c, vs, rows, S, md);
      return;
    }
    if constexpr (FS_WARP_OWNED(T, NR)) {
      for (int l = ls; l < lw; ++l)
        fw_block_level<T, NR>(Fd, l, lw, c, nsub, vs, rows, S, zsel, zt, sh.tv + (l & 1) * FS_WARPS * FS_WSL, pw, tw,
                              warp, lane);
      if (warp < nsub)
        fw_subtree<T, NR>(Fd, lw, (c << (lw - ls)) + warp, vs, rows, S, md, false, zsel, zt, pw, tw, lane);
      __syncthreads();
    }
  };
  // the levels < ls of one sweep (pass 0, or 1 for the second of mode 4) upward
  // or downward; the first one's basis rows are on their way before
  const int pstr = Fd->cap * SW_RHS_MAX;
  int buf = 0;
  auto first_level = [&](bool upward, int zsel) {
    const int l = upward ? ls - 1 : 0;
    if (ls > 0) fs_stage(Fd, l, ls, c, rkg[l], S, E - S, zsel, buf, sh);
  };
  auto global_levels = [&](bool upward, int zsel, int zt, int pass) {
    for (int q = 0; q < ls && ok; ++q) {
      const int l = upward ? ls - 1 - q : q, ln = upward ? l - 1 : l + 1;
      // the next level's copies go where the level before this one was read
      // (every thread has passed a barrier since)
      __syncthreads();
      if (q + 1 < ls) fs_stage(Fd, ln, ls, c, rkg[ln], S, E - S, zsel, buf ^ 1, sh);
      else asm volatile("cp.async.commit_group;" ::: "memory");
      ok = fs_global_level<T, NR, CL>(Fd, l, ls, c, rkg[l], vs, rows, S, E, zsel, zt,
                                  part + (size_t)(pass * ls + l) * gridDim.x * pstr, buf,
                                  bar + FS_BAR_COUNTERS + (pass << ls) + node_id(l, c >> (ls - l)), abort_flag, sh);
      buf ^= 1;
    }
    __syncthreads();
  };
  auto up = [&](int md) {  // leaves first, then the levels upward (W^-1, W^T)
    const int zsel = md == 1 ? 1 : 0, zt = md == 2 ? 1 : 0;
    first_level(true, zsel);
    local_up(md, zsel, zt);
    global_levels(true, zsel, zt, 0);
  };
  auto down = [&](int md, int pass) {  // the levels downward, then the leaves (W, W^-T)
    const int zsel = md == 3 ? 1 : 0, zt = md == 3 ? 1 : 0;
    first_level(false, zsel);
    global_levels(false, zsel, zt, pass);
    if (ok) local_down(md, zsel, zt);
  };
  if (mode == 1 || mode == 2) {
    up(mode);
  } else if (mode == 5) {  // W^-1's leaves and levels >= ls only (no CTA waits)
    local_up(1, 1, 0);
  } else if (mode == 6) {  // W^-1's levels < ls only, on v that mode 5 left
    first_level(true, 1);
    global_levels(true, 1, 0, 0);
  } else if (mode == 4) {
    up(1);
    if (ok) down(3, 1);
  } else {
    down(mode, 0);
  }
  if (!ok) return;  // the status word carries TIMEOUT; v is incomplete
  for (int j = 0; j < nrhs; ++j)
    for (int p = threadIdx.x; p < E - S; p += blockDim.x) v[(size_t)j * n + S + p] = (double)vs[(size_t)j * rows + p];
}

// Dynamic shared memory of a fused sweep.
size_t sweep_fused_smem(int rows, int nrhs, int prec);

template <typename T, int NR, bool BATCH, bool CL>
static cudaError_t launch_sweep_fused_t(cudaLaunchConfig_t& cfg, const FactDesc* Fd, double* v, int mode, int ls,
                                        int rows, double* part, unsigned int* bar, int* abort_flag,
                                        const int* active, double* const* vlist = nullptr, size_t pstride = 0) {
  const cudaError_t e = ALLOW_SMEM(k_sweep_fused<T, NR, BATCH, CL>);
  if (e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, k_sweep_fused<T, NR, BATCH, CL>, Fd, v, mode, ls, rows, part, bar, abort_flag, active,
                            vlist, pstride);
}

// ---------------------------------------------------------------------------
// Fused H-matrix product y = scale (C~ x) + shift x in one cooperative launch
// of 2^ls CTAs (the fused sweep's decomposition).  CTA c owns the rows [S, E)
// of level-ls node c: x on them sits in shared memory and each thread keeps
// the sums for its rows in registers.  The leaf blocks and the levels >= ls
// (whose nodes lie in the CTA) need nothing from other CTAs; each level < ls
// needs the projection of the partner child, which spans other CTAs.  Every CTA
// hands over its partial projections for all those levels first, works on the
// leaves and its own levels meanwhile, and then waits once for all CTAs (at a
// counter, or, launched as one cluster, at the cluster's hardware barrier) and sums
// the partner halves' partials.
//   row p in the left child of a level-l node:  y_p += U_p (V^T x_right)
//   row p in the right child:                   y_p += V_p (U^T x_left)
// (U, V share one basis array: row p holds U if p is in the left child.)
// Bound by the FP64 pipe for large n; for CTAs of few rows by how many threads
// have work, so `hs` threads share a row (leaf columns and basis columns dealt
// out between them) when there are at most 160: n = 20011, one vector, 100 -> 49
// us; n = 1000003 670 -> 626 us (0.47 ms at the FP64 peak).
// ---------------------------------------------------------------------------
#define MV_PROJ_BUF 1024                       // doubles of node projections per batch
#define MV_PART_STRIDE (FIFA_CAP_MAX * SW_RHS_MAX)  // one CTA's partial of one level
#define MV_THREADS_MAX 320

// Rows per thread, threads per row (hs) and the distance of a row's threads (rp).
struct MvShape {
  int rpt, hs, rp, threads;
};
static MvShape mv_shape(int rows) {
  if (rows <= 64) return {1, 4, 64, 256};
  if (rows <= 128) return {1, 2, 128, 256};
  if (rows <= 160) return {1, 2, 160, 320};
  int rpt = 1;
  while (rpt * 256 < rows) rpt *= 2;
  return {rpt, 1, 256, 256};
}

// BATCH: several H-matrices of one plan in one launch, problem blockIdx.y: its
// descriptor Hd[blockIdx.y], input xlist[blockIdx.y] and output ylist[...],
// its partials and its abort flag and counter (bar[0], bar[1], zeroed before)
// pstride bytes after the previous problem's (a separate instantiation:
// re-pointed arguments stay in registers).
// CL: the grid is one cluster (bar is not used then).
template <int RPT, bool BATCH = false, bool CL = false>
__global__ void __launch_bounds__(RPT == 1 ? MV_THREADS_MAX : 256, RPT <= 8 ? 4 : 2)
    k_mv_fused(const HmatDesc* __restrict__ Hd, const double* __restrict__ x, int nrhs, double* __restrict__ y, int ls,
               int rows, int hs_arg, int rp, double* __restrict__ part, unsigned int* __restrict__ bar,
               const int* __restrict__ active, const double* const* xlist, double* const* ylist, size_t pstride) {
  if (active && *active == 0) return;  // a converged iteration: nothing to compute
  if constexpr (BATCH) {
    Hd += blockIdx.y;
    x = xlist[blockIdx.y];
    y = ylist[blockIdx.y];
    part = (double*)((char*)part + blockIdx.y * pstride);
    bar = (unsigned int*)((char*)bar + blockIdx.y * pstride);
  }
  const int hs = RPT == 1 ? hs_arg : 1;
  extern __shared__ double sm[];
  double* xs = sm;                                   // nrhs x rows
  double* pj = xs + (size_t)rows * nrhs;             // MV_PROJ_BUF node projections
  double* red = pj + MV_PROJ_BUF;                    // MV_THREADS_MAX reduction partials
  int* lmap = (int*)(red + MV_THREADS_MAX);          // rows: local leaf of each row
  __shared__ int rkg[FIFA_LEVELS_MAX];               // rank of this CTA's node at each level < ls
  __shared__ int arrived;
  const int c = blockIdx.x, C = gridDim.x, tid = threadIdx.x;
  const int L = Hd->L, cap = Hd->cap, Bm = Hd->Bm;
  const int64_t n = Hd->n;
  const int* bnd = Hd->bnd;
  const int S = bnd[bnd_off(ls) + c], E = bnd[bnd_off(ls) + c + 1], R = E - S;
  const int hsel = RPT == 1 && hs > 1 ? tid / rp : 0;          // which of the row's threads
  const int row0 = RPT == 1 && hs > 1 ? tid - hsel * rp : tid;  // rows row0 + 256 i
  if (tid < ls) rkg[tid] = Hd->rank[node_id(tid, c >> (ls - tid))];
  for (int j = 0; j < nrhs; ++j)
    for (int p = tid; p < R; p += blockDim.x) xs[(size_t)j * rows + p] = x[(size_t)j * n + S + p];
  const int nl = 1 << (L - ls), first = c << (L - ls);
  for (int q = tid; q < nl; q += blockDim.x) {
    const int s0 = bnd[bnd_off(L) + first + q], e0 = bnd[bnd_off(L) + first + q + 1];
    for (int p = s0; p < e0; ++p) lmap[p - S] = q;
  }
  __syncthreads();
  // levels < ls: partial projections of this CTA's rows, w neighbouring lanes to
  // a column (few for few rows: a sum over w lanes costs log2 w additions)
  if (ls > 0) {
    const int w = R <= 256 ? 8 : (R <= 512 ? 16 : 32), ch = tid & (w - 1), ng = (int)blockDim.x / w;
    for (int l = 0; l < ls; ++l) {
      const double* Bl = Hd->bases + (size_t)l * cap * n + S;
      const int r = rkg[l];
      for (int a0 = 0; a0 < r; a0 += ng) {
        const int a = a0 + tid / w;
        double s0 = 0.0, s1 = 0.0;
        if (a < r) {
          const double* b = Bl + (size_t)a * n;
#pragma unroll 4
          for (int p = ch; p < R; p += w) {
            const double bv = b[p];
            s0 += bv * xs[p];
            if (nrhs > 1) s1 += bv * xs[rows + p];
          }
        }
        s0 = lanes_sum(s0, w);
        if (nrhs > 1) s1 = lanes_sum(s1, w);
        if (ch == 0 && a < r) {
          double* dst = part + ((size_t)c * ls + l) * MV_PART_STRIDE + a * nrhs;
          __stcg(dst, s0);
          if (nrhs > 1) __stcg(dst + 1, s1);
        }
      }
    }
    __syncthreads();
    if constexpr (CL) cluster_arrive();
    if (!CL && tid == 0) {
      __threadfence();
      atomicAdd(bar + 1, 1u);
    }
  }
  double acc[RPT][SW_RHS_MAX];
#pragma unroll
  for (int i = 0; i < RPT; ++i) acc[i][0] = acc[i][1] = 0.0;
  // leaf blocks: y_p = sum_k D[p][k] x_k over the leaf of p
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int p = S + row0 + i * 256;
    if (p < E) {
      const int q = lmap[p - S], leaf = first + q;
      const int s0 = bnd[bnd_off(L) + leaf], e0 = bnd[bnd_off(L) + leaf + 1];
      const int per = hs > 1 ? (e0 - s0 + hs - 1) / hs : e0 - s0;  // columns of each of the row's threads
      const int k0 = s0 + hsel * per, k1 = min(e0, k0 + per);
      const double* D = Hd->leaves + (size_t)leaf * Bm * Bm + (p - s0);
      double a0 = 0.0, a1 = 0.0;
      for (int k = k0; k < k1; ++k) {
        const double dv = D[(size_t)(k - s0) * Bm];
        a0 += dv * xs[k - S];
        if (nrhs > 1) a1 += dv * xs[rows + k - S];
      }
      acc[i][0] = a0;
      acc[i][1] = a1;
    }
  }
  // levels >= ls: nodes inside this CTA, in batches whose projections fit pj
  for (int l = ls; l < L; ++l) {
    const double* Bl = Hd->bases + (size_t)l * cap * n;
    const int nsub = 1 << (l - ls), i0 = c << (l - ls);
    int rmax = 0;
    for (int q = 0; q < nsub; ++q) rmax = max(rmax, Hd->rank[node_id(l, i0 + q)]);
    if (rmax == 0) continue;
    const int per = 2 * rmax * nrhs;  // projection entries per node: (side, c, j)
    const int nb = max(1, MV_PROJ_BUF / per);
    for (int b0 = 0; b0 < nsub; b0 += nb) {
      const int bn = min(nb, nsub - b0);
      tile_dots(bn * per, Bl, n, xs, rows, S,
              [&](int o, int& a0, int& a1, int& col, int& j) {
                const int node = o / per, rem = o % per, side = rem / (rmax * nrhs), cj = rem % (rmax * nrhs);
                const int cc = cj / nrhs;
                j = cj % nrhs;
                const int nid = node_id(l, i0 + b0 + node);
                int s0, h0, e0;
                node_range(bnd, l, i0 + b0 + node, s0, h0, e0);
                a0 = side ? h0 : s0;
                a1 = side ? e0 : h0;
                col = cc < Hd->rank[nid] ? cc : -1;
              },
              red, pj);
      // rows of the batch's nodes: y_p += basis_l[p] . proj(partner side)
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        const int p = S + row0 + i * 256;
        if (p < E) {
          const int node = (lmap[p - S] >> (L - l)) - b0;
          if (node >= 0 && node < bn) {
            const int gi = i0 + b0 + node;
            const int r = Hd->rank[node_id(l, gi)];
            int s0, h0, e0;
            node_range(bnd, l, gi, s0, h0, e0);
            const int other = p < h0 ? 1 : 0;
            const double* pr = pj + node * per + other * rmax * nrhs;
            double a0 = acc[i][0], a1 = acc[i][1];  // products accumulate onto the row sums
            for (int cc = hsel; cc < r; cc += hs) {
              const double bv = Bl[(size_t)cc * n + p];
              a0 += bv * pr[cc * nrhs];
              if (nrhs > 1) a1 += bv * pr[cc * nrhs + 1];
            }
            acc[i][0] = a0;
            acc[i][1] = a1;
          }
        }
      }
      __syncthreads();
    }
  }
  if (ls > 0) {
    // every CTA's partials are written (a bounded wait; a launch's CTAs are all resident)
    if constexpr (CL) {
      __syncthreads();
      cluster_wait();
    }
    if (!CL && tid == 0) {
      volatile int* abort_flag = (volatile int*)bar;
      const unsigned int limit = Hd->spin ? Hd->spin : FIFA_SPIN_LIMIT;
      unsigned int spins = 0;
      int ok = 1;
      while (*((volatile unsigned int*)(bar + 1)) < (unsigned)C) {
        if (*abort_flag) {
          ok = 0;
          break;
        }
        if (++spins > limit) {
          atomicOr(Hd->status, FIFA_DEV_TIMEOUT);
          *abort_flag = 1;
          ok = 0;
          break;
        }
        if (spins > 256) __nanosleep(64);
      }
      __threadfence();
      arrived = ok;
    }
    if constexpr (!CL) {
      __syncthreads();
      if (!arrived) return;
    }
  }
  // levels < ls, as many at a time as fit pj: the partner halves' projections,
  // then the rows' sums
#pragma unroll 1
  for (int l0 = 0; l0 < ls;) {
    int l1 = l0, tot = 0;
    while (l1 < ls && tot + rkg[l1] * nrhs <= MV_PROJ_BUF) tot += rkg[l1++] * nrhs;
    int off = 0;
    for (int l = l0; l < l1; ++l) {
      const int span = ls - l, i = c >> span, side = (c >> (span - 1)) & 1;
      const int K = rkg[l] * nrhs, half = 1 << (span - 1);
      const int c0 = (i << span) + (1 - side) * half;  // first CTA of the partner child
      const int w = min(half, 32), ch = tid & (w - 1), ng = (int)blockDim.x / w;
      for (int o0 = 0; o0 < K; o0 += ng) {
        const int k = o0 + tid / w;
        double v = 0.0;
        if (k < K) {
          const double* src = part + ((size_t)c0 * ls + l) * MV_PART_STRIDE + k;
#pragma unroll 8
          for (int q = ch; q < half; q += w) v += __ldcg(src + (size_t)q * ls * MV_PART_STRIDE);
        }
        v = lanes_sum(v, w);
        if (ch == 0 && k < K) pj[off + k] = v;
      }
      off += K;
    }
    __syncthreads();
#pragma unroll
    for (int ii = 0; ii < RPT; ++ii) {
      const int p = S + row0 + ii * 256;
      if (p < E) {
        double a0 = acc[ii][0], a1 = acc[ii][1];
        const double* pr = pj;
        for (int l = l0; l < l1; ++l) {
          const double* Bl = Hd->bases + (size_t)l * cap * n + p;
          const int r = rkg[l];
          for (int cc = hsel; cc < r; cc += hs) {
            const double bv = Bl[(size_t)cc * n];
            a0 += bv * pr[cc * nrhs];
            if (nrhs > 1) a1 += bv * pr[cc * nrhs + 1];
          }
          pr += r * nrhs;
        }
        acc[ii][0] = a0;
        acc[ii][1] = a1;
      }
    }
    __syncthreads();
    l0 = l1;
  }
  if (RPT == 1 && hs > 1) {  // the row's threads together, in order
    if (hsel > 0 && S + row0 < E) {
      pj[((hsel - 1) * rp + row0) * 2] = acc[0][0];
      pj[((hsel - 1) * rp + row0) * 2 + 1] = acc[0][1];
    }
    __syncthreads();
    if (hsel > 0) return;
    if (S + row0 < E)
      for (int q = 0; q < hs - 1; ++q) {
        acc[0][0] += pj[(q * rp + row0) * 2];
        acc[0][1] += pj[(q * rp + row0) * 2 + 1];
      }
  }
  const double sc = Hd->scale, shf = Hd->shift;
  const double* dg = Hd->diag;
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int p = S + row0 + i * 256;
    if (p < E) {
      const bool plain = !dg && shf == 0.0 && sc == 1.0;
      const double sh = dg ? dg[p] : shf;
      y[p] = plain ? acc[i][0] : sc * acc[i][0] + sh * xs[p - S];
      if (nrhs > 1) y[n + p] = plain ? acc[i][1] : sc * acc[i][1] + sh * xs[rows + p - S];
    }
  }
}

size_t mv_fused_smem(int rows);

template <int RPT, bool BATCH, bool CL>
static cudaError_t launch_mv_fused_t(const HmatDesc* Hd, int ls, int rows, const double* x, int nrhs, double* y,
                                     double* part, unsigned int* bar, cudaStream_t st, const int* active,
                                     const double* const* xlist = nullptr, double* const* ylist = nullptr,
                                     int nprob = 1, size_t pstride = 0) {
  const size_t smem = mv_fused_smem(rows);
  const MvShape sh = mv_shape(rows);
  const cudaError_t e = ALLOW_SMEM(k_mv_fused<RPT, BATCH, CL>);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1u << ls, nprob);
  cfg.blockDim = dim3(sh.threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  if (CL) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1u << ls;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
  } else {
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_mv_fused<RPT, BATCH, CL>, Hd, x, nrhs, y, ls, rows, sh.hs, sh.rp, part, bar, active,
                            xlist, ylist, pstride);
}

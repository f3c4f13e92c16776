// Level kernel of the factorization for ranks <= 16: one tree node by one CTA,
// by a thread-block cluster, or (large nodes) by a group of CTAs that meet at
// bounded-spin barriers; the node's rows are split evenly over the CTAs.
//
// Per node (X the r basis columns of both sides, B the ancestor columns on the
// node's rows; all sums over rows exchanged between the node's CTAs):
//   1. Gram(X);  R1 = chol, Q1 = X R1^-1 (each side alone)
//   2. Gram(Q1) = I + E and P1 = Q1^T B together;  R2 = chol(I + E), R = R2 R1,
//      P = R2^-T P1 = Q^T B.  E is rounding (u times the squared condition number
//      of the column-scaled X), so R2 = I + F + O(E^2) with F the strict upper
//      triangle and half the diagonal of E: no chain of pivots.  Above
//      ND_E_MAX, where E^2 would show, R2 is factored like R1.
//   3. S = I + R X R^T = [I M; M^T I], M = R_U R_V^T, so L_S = [I 0; M^T L2] with
//      L2 = chol(I - M^T M) and L_S^-1 = [I 0; K L2^-1], K = -L2^-1 M^T: r pivots
//      instead of 2r, and T = (L_S^-1 - I) P is zero on the left side, whose rows
//      of B keep their values.
//   4. B_right += Q1 (R2^-1 T);  Q = Q1 R2^-1
// so a level costs two exchanges however many ancestor columns it has (more
// only beyond a buffer's worth of them): the small dense algebra is repeated by
// every CTA, which reads the same sums and so finds the same bits.
//
// What bounds it: small nodes the serial chain of the small algebra (a dependent
// FP64 instruction takes a warp 64 cycles, an instruction fetched for the first
// time several hundred), large ones the FP64 pipe (2 lanes per cycle and SM).
// Hence the elimination by one warp with few FP64 instructions per pivot, loops
// rather than unrolled code, and, where a CTA's rows and columns fit the
// row tiles, all of them resident in shared memory from one load to one store.
// Against three exchanges and more per level, one-thread algebra and an update of
// both sides: a level of n = 2048 (64-row leaves, ranks to 14) 128-189 -> 33-80
// us; one factorization of n = 2^20 (clustered inputs, ranks 2 to 7) 11.8 -> 10.6
// ms with the leaf factor's changes, its levels at 45-68% of the FP64 peak.
#include <algorithm>
#include <atomic>

#include "fifa_common.cuh"
#include "fifa_launch.h"
#include "fifa_level.cuh"

#define ND_W 8     // ancestor columns per staged tile
#define ND_CW 24   // ancestor columns per exchange at rank RB (more at lower ranks)
#define ND_COLS 128  // most ancestor columns per exchange
#define ND_E_MAX 0x1p-30  // r E^2 then stays below 2^-56

template <int RB>
struct NdLayout {
  static constexpr int mat = RB * RB;
  static constexpr int xn = RB * (RB + 1) + 2 * RB * ND_CW;   // one exchange: packed Gram of both sides, 2r x columns
  static constexpr int tbuf = (RB + ND_W) * LV_TRP;           // doubles per row tile
  static constexpr int fixed = 7 * mat + 2 * RB + xn + 2 * tbuf + 256 + 4;
  static size_t bytes(int cluster) {
    return (size_t)(fixed + (cluster > 1 ? 2 * xn : 0)) * sizeof(double) + ND_COLS * sizeof(double*) +
           (FIFA_LEVELS_MAX + 4) * sizeof(int);
  }
};

// Load a double of the same shared-memory variable in CTA `rank` of the cluster.
__device__ __forceinline__ double ld_cluster(const double* p, int rank) {
  unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
  double v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(r) : "memory");
  return v;
}

// Pairs of columns in shared memory (column c at src + c ld): out[idx(o)] = sum
// over local rows [a0, a1) of column ca times column cb, o -> (ca, cb) by pair().
template <typename PairF, typename IdxF>
__device__ void smem_pairs(const double* src, int ld, int np_all, int a0, int a1, double* part, double* out, PairF pair,
                           IdxF idx) {
  const int t = threadIdx.x;
  if (a1 <= a0) {
    for (int q = t; q < np_all; q += blockDim.x) out[idx(q)] = 0.0;
    return;
  }
  for (int q0 = 0; q0 < np_all; q0 += blockDim.x) {
    const int np = min((int)blockDim.x, np_all - q0);
    const int ng = min((int)blockDim.x / np, 8);
    const bool active = t < np * ng;
    const int o = active ? t % np : 0, gidx = active ? t / np : 0;
    int ca, cb;
    pair(q0 + o, ca, cb);
    const double* ta = src + ca * ld;
    const double* tb = src + cb * ld;
    double s0 = 0.0, s1 = 0.0;
    if (active) {
      int p = a0 + gidx;
      for (; p + ng < a1; p += 2 * ng) {
        s0 += ta[p] * tb[p];
        s1 += ta[p + ng] * tb[p + ng];
      }
      if (p < a1) s0 += ta[p] * tb[p];
    }
    s0 += s1;
    if (ng == 1) {
      if (active) out[idx(q0 + o)] = s0;
      continue;
    }
    if (active) part[gidx * np + o] = s0;
    __syncthreads();
    if (t < np) {
      double v = part[t];
      for (int w = 1; w < ng; ++w) v += part[w * np + t];
      out[idx(q0 + t)] = v;
    }
    __syncthreads();
  }
}

// out[idx(o)] = sum over rows [a0, a1) of col(ca)[p] * col(cb)[p] for the np_all
// outputs o -> (ca, cb) of pair(); the ncol columns are staged tile by tile.
template <typename ColF, typename PairF, typename IdxF>
__device__ void tile_pairs(double* tile, int tbuf, int ncol, int np_all, int a0, int a1, double* part, double* out,
                           ColF col, PairF pair, IdxF idx) {
  const int t = threadIdx.x;
  if (a1 <= a0) {
    for (int q = t; q < np_all; q += blockDim.x) out[idx(q)] = 0.0;
    return;
  }
  for (int q0 = 0; q0 < np_all; q0 += blockDim.x) {
    const int np = min((int)blockDim.x, np_all - q0);
    const int ng = (int)blockDim.x / np;
    const bool active = t < np * ng;
    const int o = active ? t % np : 0, gidx = active ? t / np : 0;
    int ca, cb;
    pair(q0 + o, ca, cb);
    double acc = 0.0;
    tile_walk<double>(tile, tbuf, ncol, a0, a1, col, [&](const double* tl, int tr) {
      if (active) {
        const double* ta = tl + ca * LV_TRP;
        const double* tb = tl + cb * LV_TRP;
#pragma unroll 4
        for (int p = gidx; p < tr; p += ng) acc += ta[p] * tb[p];
      }
    });
    if (ng == 1) {
      if (active) out[idx(q0 + o)] = acc;
      continue;
    }
    if (active) part[gidx * np + o] = acc;
    __syncthreads();
    for (int w = ng; w > 1;) {  // pairwise tree over the ng partials of every output
      const int hw = (w + 1) / 2;
      for (int i = t; i < (w - hw) * np; i += blockDim.x) part[i] += part[i + hw * np];
      w = hw;
      __syncthreads();
    }
    for (int q = t; q < np; q += blockDim.x) out[idx(q0 + q)] = part[q];
    __syncthreads();
  }
}

// Rows [a0, a1): X[:, p] <- X[:, p] Ri with Ri = Li^T (Li lower, rows RB apart).
template <int RB>
__device__ void rowmul(double* __restrict__ Xb, int64_t n, int r, int a0, int a1, const double* Li) {
  for (int p = a0 + threadIdx.x; p < a1; p += blockDim.x) {
    double x[RB];
#pragma unroll
    for (int c = 0; c < RB; ++c)
      if (c < r) x[c] = Xb[(size_t)c * n + p];
#pragma unroll
    for (int c = 0; c < RB; ++c)
      if (c < r) {
        double v = 0.0;
#pragma unroll
        for (int a = 0; a <= c; ++a) v += x[a] * Li[c * RB + a];
        Xb[(size_t)c * n + p] = v;
      }
  }
}

// Rows [a0, a1): B_j[p] += sum_a Q[a][p] T[a * ldt + j] for w columns, eight at
// a time; a CTA with few rows spreads the column chunks over its thread groups.
template <int RB>
__device__ void col_update(const double* __restrict__ Qb, double* const* Bp, int64_t n, int r, int w, int a0, int a1,
                           const double* T, int ldt) {
  const int rows = a1 - a0;
  if (rows <= 0) return;
  const int span = min((rows + 31) & ~31, (int)blockDim.x), nsub = (int)blockDim.x / span;
  const int sub = threadIdx.x / span, pt = threadIdx.x % span;
  if (sub >= nsub) return;
  for (int j0 = sub * ND_W; j0 < w; j0 += nsub * ND_W) {
    const int wn = min(ND_W, w - j0);
    for (int p = a0 + pt; p < a1; p += span) {
      double acc[ND_W];
#pragma unroll
      for (int j = 0; j < ND_W; ++j)
        if (j < wn) acc[j] = Bp[j0 + j][p];
      for (int a = 0; a < r; ++a) {
        const double q = Qb[(size_t)a * n + p];
#pragma unroll
        for (int j = 0; j < ND_W; ++j)
          if (j < wn) acc[j] += q * T[a * ldt + j0 + j];
      }
#pragma unroll
      for (int j = 0; j < ND_W; ++j)
        if (j < wn) Bp[j0 + j][p] = acc[j];
    }
  }
}

// RB: largest rank taken, RLO: ranks up to it are another launch's (-1: all).
// CL: the G CTAs of a node are a thread-block cluster (G = 1: a CTA alone) and
// exchange through distributed shared memory; else a group of co-resident CTAs
// of a cooperative launch.
template <int RB, int RLO, bool CL>
__global__ void __launch_bounds__(256, RB == 4 ? 4 : 3)
    k_level(const FactDesc* __restrict__ Fd, int lvl, int G, double* __restrict__ gpart,
            unsigned int* __restrict__ bar, int* __restrict__ abort_flag, int skip_le, size_t sstride) {
  extern __shared__ double sm[];
  using LY = NdLayout<RB>;
  Fd += blockIdx.y;  // problem of a batched launch: its descriptor, and its scratch sstride bytes on
  if (Fd->skip && *Fd->skip) return;  // the same for every CTA: none waits on a missing one
  gpart = (double*)((char*)gpart + blockIdx.y * sstride);
  bar = (unsigned int*)((char*)bar + blockIdx.y * sstride);
  abort_flag = (int*)((char*)abort_flag + blockIdx.y * sstride);
  const int bi = blockIdx.x / G, g = blockIdx.x % G, base = blockIdx.x - g;
  const int nid = node_id(lvl, bi);
  const int r = Fd->rank[nid];
  if (r <= skip_le || r <= RLO || r > RB) return;  // another launch takes this node
  const int cap = Fd->cap, nleaf = Fd->nleaf;
  const int64_t n = Fd->n;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int s, h, e;
  node_range(Fd->bnd, lvl, bi, s, h, e);
  if (r == 0) {
    if (g == 0 && tid == 0) Fd->ld_parts[nleaf + nid] = 0.0;
    return;
  }
  double* Qall = (double*)Fd->Q;
  double* Qb = Qall + (size_t)lvl * cap * n;

  double* M1 = sm;                     // Gram / factor of both sides (RB x RB each), then I - M^T M / L2 and K
  double* RU = M1 + 2 * LY::mat;       // R = R2 R1 of both sides
  double* Li = RU + 2 * LY::mat;       // R2^-T of both sides
  double* Mm = Li + 2 * LY::mat;       // M = R_U R_V^T
  double* Rd = Mm + LY::mat;           // diagonals of the two factors
  double* xs = Rd + 2 * RB;            // sums of an exchange: packed Gram left, right, then 2r x cw
  double* tile = xs + LY::xn;          // two row tiles, or this CTA's rows of X and of an exchange's columns
  double* part = tile + 2 * LY::tbuf;  // 256 partial sums
  double* xb = part + 256 + 4;         // cluster: two exchange buffers
  double** Bp = (double**)(xb + (CL && G > 1 ? 2 * LY::xn : 0));  // an exchange's columns
  int* apre = (int*)(Bp + ND_COLS);    // prefix sums of the ancestor ranks
  int* iflag = apre + FIFA_LEVELS_MAX + 1;  // [0] a pivot failed, [1] |E| above ND_E_MAX
  const int npk = r * (r + 1) / 2;
  const size_t pstride = level_part_stride(cap);
  unsigned int phase = 0;

  if (warp == 0) {
    int c = lane < lvl ? Fd->rank[node_id(lane, bi >> (lvl - lane))] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, c, o);
      if (lane >= o) c += t;
    }
    if (lane < lvl) apre[lane + 1] = c;
    if (lane == 0) {
      apre[0] = 0;
      iflag[0] = iflag[1] = 0;
    }
  }
  __syncthreads();
  const int na = apre[lvl];
  const int len = e - s, rc = (len + G - 1) / G;
  const int r0 = s + min(len, g * rc), r1 = s + min(len, g * rc + rc);
  const int sa0 = r0, sa1 = max(r0, min(r1, h)), sb0 = max(min(r1, h), r0), sb1 = r1;  // its rows of the two sides

  // columns of an exchange, and whether they and X fit the row tiles
  const int cwmax = min(min((2 * RB * ND_CW) / (2 * r), ND_COLS), CL ? ND_COLS : ((int)pstride - 2 * npk) / (2 * r));
  int cw = min(na, cwmax);
  if (cw < na && cw > ND_W) cw -= cw % ND_W;
  const int rows = r1 - r0, ld = rows | 1;
  const bool res = (long long)(r + cw) * ld <= 2 * LY::tbuf;
  auto columns = [&](int c0, int w) {  // pointers of ancestor columns [c0, c0 + w)
    for (int t = tid; t < w; t += blockDim.x) {
      const int c = c0 + t;
      int j = 0;
      while (apre[j + 1] <= c) ++j;
      Bp[t] = Qall + ((size_t)j * cap + (c - apre[j])) * n;
    }
    __syncthreads();
  };
  auto stage_b = [&](int w) {  // this CTA's rows of the columns, behind X (asynchronous)
    for (int i = tid; i < w * rows; i += blockDim.x) {
      const int c = i / rows, p = i - c * rows;
      cp_async8(tile + (r + c) * ld + p, Bp[c] + r0 + p);
    }
    cp_async_commit();
  };

  // sum `count` doubles of every CTA of the node: each puts its own at slot()
  // before, all find the sums in xs after
  auto slot = [&]() -> double* { return CL && G > 1 ? xb + (phase & 1u) * LY::xn : xs; };
  auto exchange = [&](int count) -> bool {
    __syncthreads();
    if (G == 1) return true;
    if constexpr (CL) {
      // two buffers in turn: one is written again only after the next barrier,
      // which every reader of its previous contents has passed
      const double* mine = slot();
      cluster_sync_all();
      for (int t = tid; t < count; t += blockDim.x) {
        double sum = 0.0;
        for (int q0 = 0; q0 < G; q0 += 8) {
          double v[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) v[q] = q0 + q < G ? ld_cluster(mine + t, q0 + q) : 0.0;
#pragma unroll
          for (int o = 4; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (q < o) v[q] += v[q + o];
          sum += v[0];
        }
        xs[t] = sum;
      }
      ++phase;
      __syncthreads();
      return true;
    } else {
      return group_reduce(xs, xs, count, G, g, base, gpart, pstride, bar, phase, Fd->status, abort_flag, part, Fd->spin);
    }
  };
  auto gram_pair = [&](int o, int& a, int& b) { pair_decode(o, r, a, b); };
  auto xcol = [&](int c) -> const double* { return Qb + (size_t)c * n; };

  columns(0, cw);
  if (res) {
    for (int i = tid; i < r * rows; i += blockDim.x) {
      const int c = i / rows, p = i - c * rows;
      cp_async8(tile + c * ld + p, Qb + (size_t)c * n + r0 + p);
    }
    cp_async_commit();
    stage_b(cw);
    cp_async_wait_prev();  // X is here, B may still be on its way
    __syncthreads();
  }
  // X[:, p] <- X[:, p] Ri on this CTA's rows, Ri^T the lower triangles Lm, Lm + mat
  auto rows_times = [&](const double* Lm) {
    if (res) {
      // a warp per 32 rows and column, columns from the right: a round's
      // columns are stored after all of its sums have been taken, and later
      // rounds read only columns further left
      const int nblk = (rows + 31) / 32, nw = (int)blockDim.x >> 5;
      for (int u0 = 0; u0 < r * nblk; u0 += nw) {
        const int u = u0 + warp, c = r - 1 - u / nblk, p = (u % nblk) * 32 + lane;
        double v = 0.0;
        if (u < r * nblk && p < rows) {
          const double* Ls = Lm + (r0 + p < h ? 0 : LY::mat) + c * RB;
          const double* x = tile + p;
          for (int a = 0; a <= c; ++a) v += x[a * ld] * Ls[a];
        }
        __syncthreads();
        if (u < r * nblk && p < rows) tile[c * ld + p] = v;
      }
    } else {
      rowmul<RB>(Qb, n, r, sa0, sa1, Lm);
      rowmul<RB>(Qb, n, r, sb0, sb1, Lm + LY::mat);
    }
    __syncthreads();
  };
  // P[a][j] (rows of the left side a < r, of the right r <= a) for w columns
  // behind ng Gram entries of each side, to dst
  auto project = [&](int w, double* dst, int ng) {
    for (int sd = 0; sd < 2; ++sd) {
      const int a0 = sd ? sb0 : sa0, a1 = sd ? sb1 : sa1;
      const int wstep = res ? max(w, 1) : ND_W;
      int j0 = 0;
      do {
        const int wn = min(wstep, w - j0), gr = j0 == 0 ? ng : 0;
        auto pair = [&](int o, int& a, int& b) {
          if (o < gr) {
            pair_decode(o, r, a, b);
          } else {
            a = (o - gr) / wn;
            b = r + (o - gr) % wn;
          }
        };
        auto idx = [&](int o) {
          return o < gr ? sd * ng + o : 2 * ng + (sd * r + (o - gr) / wn) * w + j0 + (o - gr) % wn;
        };
        if (res)
          smem_pairs(tile, ld, gr + r * wn, a0 - r0, a1 - r0, part, dst, pair, idx);
        else
          tile_pairs(tile, LY::tbuf, r + wn, gr + r * wn, a0, a1, part, dst,
                     [&](int c) -> const double* { return c < r ? Qb + (size_t)c * n : Bp[j0 + c - r]; }, pair, idx);
        j0 += wstep;
      } while (j0 < w);
    }
  };

  // 1. Gram(X), R1, Q1 = X R1^-1
  project(0, slot(), npk);
  if (!exchange(2 * npk)) return;
  auto unpack = [&](double* G2) {  // both sides' Gram sums (upper triangles)
    for (int q = tid; q < 2 * npk; q += blockDim.x) {
      const int sd = q >= npk;
      int a, b;
      pair_decode(q - sd * npk, r, a, b);
      G2[sd * LY::mat + a * RB + b] = xs[q];
    }
    __syncthreads();
  };
  unpack(M1);
  if (warp < 2 && !warp_chol_inv(M1 + warp * LY::mat, RB, r, Rd + warp * RB, lane) && lane == 0) iflag[0] = 1;
  __syncthreads();
  rows_times(M1);

  // 2. Gram(Q1) and P1 = Q1^T B
  cp_async_wait_all();
  __syncthreads();
  project(cw, slot(), npk);
  if (!exchange(2 * npk + 2 * r * cw)) return;
  // E and F; R2^-T = I - F^T and R = R1 + F R1, or R2 factored
  for (int q = tid; q < 2 * npk; q += blockDim.x) {
    const int sd = q >= npk;
    int a, b;
    pair_decode(q - sd * npk, r, a, b);
    const double E = xs[q] - (a == b ? 1.0 : 0.0);
    if (!(fabs(E) <= ND_E_MAX)) iflag[1] = 1;
    Li[sd * LY::mat + b * RB + a] = a == b ? 1.0 - 0.5 * E : -E;
  }
  __syncthreads();
  const bool full = iflag[1] != 0;  // from the same sums in every CTA
  if (full) {
    unpack(Li);
    if (warp < 2 && !warp_chol_inv(Li + warp * LY::mat, RB, r, part + warp * RB, lane) && lane == 0) iflag[0] = 1;
    __syncthreads();
  }
  for (int t = tid; t < 2 * r * r; t += blockDim.x) {
    const int sd = t >= r * r, q = t - sd * r * r, i = q / r, j = q % r;
    if (i > j) continue;
    const double* R1 = M1 + sd * LY::mat;
    const double* Rdd = Rd + sd * RB;
    const double* L2m = Li + sd * LY::mat;
    // R2[i][k] is F = -(R2^-T)[k][i] off the diagonal in the first-order case
    double v = (full ? part[sd * RB + i] : 2.0 - L2m[i * RB + i]) * (i == j ? Rdd[j] : R1[i * RB + j]);
    for (int k = i + 1; k <= j; ++k)
      v += (full ? L2m[i * RB + k] : -L2m[k * RB + i]) * (k == j ? Rdd[j] : R1[k * RB + j]);
    RU[sd * LY::mat + i * RB + j] = v;
  }
  __syncthreads();
  // 3. M = R_U R_V^T, I - M^T M = L2 L2^T; meanwhile P = R2^-T P1
  for (int t = tid; t < r * r; t += blockDim.x) {
    const int a = t / r, b = t % r;
    double v = 0.0;
    for (int k = max(a, b); k < r; ++k) v += RU[a * RB + k] * RU[LY::mat + b * RB + k];
    Mm[a * RB + b] = v;
  }
  __syncthreads();
  for (int t = tid; t < r * r; t += blockDim.x) {
    const int a = t / r, b = t % r;
    if (a > b) continue;
    double v = a == b ? 1.0 : 0.0;
    for (int k = 0; k < r; ++k) v -= Mm[k * RB + a] * Mm[k * RB + b];
    M1[a * RB + b] = v;
  }
  double* Pm = xs + 2 * npk;
  __syncthreads();
  if (warp == 0) {
    if (!warp_chol_inv(M1, RB, r, Rd, lane) && lane == 0) iflag[0] = 1;
  } else {
    for (int t = tid - 32; t < 2 * cw; t += blockDim.x - 32) {  // a thread per side and column, rows from the bottom
      const int sd = t >= cw, j = sd ? t - cw : t;
      const double* Ls = Li + sd * LY::mat;
      double* Pc = Pm + (size_t)sd * r * cw + j;
      for (int a = r - 1; a >= 0; --a) {
        double v = 0.0;
        for (int b = 0; b <= a; ++b) v += Ls[a * RB + b] * Pc[b * cw];
        Pc[a * cw] = v;
      }
    }
  }
  __syncthreads();
  // K = -L2^-1 M^T
  double* K = M1 + LY::mat;
  for (int t = tid; t < r * r; t += blockDim.x) {
    const int a = t / r, c = t % r;
    double v = 0.0;
    for (int b = 0; b <= a; ++b) v -= M1[a * RB + b] * Mm[c * RB + b];
    K[a * RB + c] = v;
  }
  __syncthreads();
  if (g == 0) {
    const int ld2 = 2 * cap, r2 = 2 * r;
    double* Zf = Fd->Zf + (size_t)nid * ld2 * ld2;
    double* Zi = Fd->Zi + (size_t)nid * ld2 * ld2;
    for (int t = tid; t < r2 * r2; t += blockDim.x) {
      const int a = t / r2, b = t % r2, ra = a - r, rb = b - r;
      double zf = 0.0, zi = 0.0;
      if (ra >= 0 && rb < 0) {
        zf = Mm[b * RB + ra];
        zi = K[ra * RB + b];
      } else if (ra >= 0 && rb <= ra) {
        zf = ra == rb ? Rd[ra] - 1.0 : M1[rb * RB + ra];
        zi = M1[ra * RB + rb] - (ra == rb ? 1.0 : 0.0);
      }
      Zf[a * ld2 + b] = zf;
      Zi[a * ld2 + b] = zi;
    }
    if (warp == 7) {
      double ls = lane < r ? log(Rd[lane]) : 0.0;
      ls = warp_sum(ls);
      if (lane == 0) {
        Fd->ld_parts[nleaf + nid] = ls;
        if (iflag[0]) atomicOr(Fd->status, FIFA_DEV_NOT_SPD);
      }
    }
  }
  // 4. T = K P_left + (L2^-1 - I) P_right over P_left's place (at most two
  // entries per thread); for the first columns R2^-1 T, since the rows still hold Q1
  static_assert(RB * ND_CW <= 2 * 256, "two entries of T per thread");
  auto put2 = [&](int cnt, auto val) {
    double v0 = 0.0, v1 = 0.0;
    if (tid < cnt) v0 = val(tid);
    if (tid + 256 < cnt) v1 = val(tid + 256);
    __syncthreads();
    if (tid < cnt) Pm[tid] = v0;
    if (tid + 256 < cnt) Pm[tid + 256] = v1;
    __syncthreads();
  };
  auto update = [&](int w, bool first) {
    const double* Pr = Pm + (size_t)r * w;
    put2(r * w, [&](int t) {
      const int a = t / w, j = t % w;
      double v0 = (M1[a * RB + a] - 1.0) * Pr[a * w + j], v1 = 0.0;
      for (int b = 0; b < a; ++b) v0 += M1[a * RB + b] * Pr[b * w + j];
      for (int b = 0; b < r; ++b) v1 += K[a * RB + b] * Pm[b * w + j];
      return v0 + v1;
    });
    if (first)
      put2(r * w, [&](int t) {
        const int a = t / w, j = t % w;
        double v = 0.0;
        for (int b = a; b < r; ++b) v += Li[LY::mat + b * RB + a] * Pm[b * w + j];
        return v;
      });
    if (res) {
      const int nr = sb1 - sb0, p0 = sb0 - r0;
      for (int i = tid; i < nr * w; i += blockDim.x) {
        const int j = i / nr, p = p0 + i - j * nr;
        double v0 = tile[(r + j) * ld + p], v1 = 0.0;
        int a = 0;
        for (; a + 1 < r; a += 2) {
          v0 += tile[a * ld + p] * Pm[a * w + j];
          v1 += tile[(a + 1) * ld + p] * Pm[(a + 1) * w + j];
        }
        if (a < r) v0 += tile[a * ld + p] * Pm[a * w + j];
        Bp[j][r0 + p] = v0 + v1;
      }
    } else {
      col_update<RB>(Qb, Bp, n, r, w, sb0, sb1, Pm, w);
    }
    __syncthreads();
  };
  if (cw > 0) update(cw, true);
  rows_times(Li);
  if (res)
    for (int i = tid; i < r * rows; i += blockDim.x) {
      const int c = i / rows, p = i - c * rows;
      Qb[(size_t)c * n + r0 + p] = tile[c * ld + p];
    }
  // further ancestor columns, with Q in place
  for (int c0 = cw; c0 < na; c0 += cw) {
    const int w = min(cw, na - c0);
    columns(c0, w);
    if (res) {
      stage_b(w);
      cp_async_wait_all();
      __syncthreads();
    }
    Pm = xs;
    project(w, slot(), 0);
    if (!exchange(2 * r * w)) return;
    update(w, false);
  }
  if (CL && G > 1) cluster_sync_all();  // no CTA leaves while another may still read its sums
}

// ---------------------------------------------------------------------------
// Host launchers.
// ---------------------------------------------------------------------------
template <int RB, int RLO, bool CL>
static cudaError_t launch_node_t(const FactDesc* Fd, int lvl, int nodes, int G, double* part, unsigned int* bar,
                                 int* abort_flag, int skip, cudaStream_t st, int nprob, size_t sstride) {
  const size_t smem = NdLayout<RB>::bytes(CL ? G : 1);
  const cudaError_t e = ALLOW_SMEM(k_level<RB, RLO, CL>);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nodes * G, nprob);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  if (CL) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = G;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
  } else {
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = G > 1 ? 1 : 0;
  }
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_level<RB, RLO, CL>, Fd, lvl, G, part, bar, abort_flag, skip, sstride);
}

cudaError_t launch_node(const FactDesc* Fd, int rb, int rlo, bool cluster, int lvl, int nodes, int G, double* part,
                        unsigned int* bar, int* abort_flag, int skip, cudaStream_t st, int nprob, size_t sstride) {
#define ND_GO(RB, RLO)                                                                                          \
  return cluster ? launch_node_t<RB, RLO, true>(Fd, lvl, nodes, G, part, bar, abort_flag, skip, st, nprob, sstride) \
                 : launch_node_t<RB, RLO, false>(Fd, lvl, nodes, G, part, bar, abort_flag, skip, st, nprob, sstride)
  if (rb == 4) ND_GO(4, -1);
  if (rlo >= 4) ND_GO(16, 4);
  ND_GO(16, -1);
#undef ND_GO
}

// Largest cluster of the level kernels: 16 CTAs, beyond the portable eight,
// where the GPU can hold one.
template <int RB, int RLO>
static bool node_cluster16() {
  const size_t smem = NdLayout<RB>::bytes(16);
  if (ALLOW_SMEM(k_level<RB, RLO, true>) != cudaSuccess ||
      cudaFuncSetAttribute(k_level<RB, RLO, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    return false;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(16);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 16;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int held = 0;
  return cudaOccupancyMaxActiveClusters(&held, k_level<RB, RLO, true>, &cfg) == cudaSuccess && held > 0;
}
// (for the current device: the permission that node_cluster16 sets is the
// device's own, as is the answer)
int node_cluster_max() {
  static std::atomic<unsigned long long> asked{0}, sixteen{0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 8;
  const unsigned long long bit = 1ull << (dev & 63);
  if (!(asked.load(std::memory_order_acquire) & bit)) {
    if (node_cluster16<4, -1>() && node_cluster16<16, 4>() && node_cluster16<16, -1>()) sixteen.fetch_or(bit);
    cudaGetLastError();
    asked.fetch_or(bit, std::memory_order_release);
  }
  return sixteen.load(std::memory_order_relaxed) & bit ? 16 : 8;
}

template <int RB, int RLO>
static int node_per_sm() {
  const size_t smem = NdLayout<RB>::bytes(1);
  ALLOW_SMEM(k_level<RB, RLO, false>);
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_level<RB, RLO, false>, 256, smem) != cudaSuccess) per_sm = 0;
  cudaGetLastError();
  return per_sm;
}
int node_ctas_per_sm(int rb) { return rb == 4 ? node_per_sm<4, -1>() : std::min(node_per_sm<16, 4>(), node_per_sm<16, -1>()); }

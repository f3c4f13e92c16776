// Application kernels: W, W^T, W^-1, W^-T sweeps (SI: W = A_L ... A_0 with
// node factors I + Q Z Q^T) and the H-matrix product (leaf products plus the
// low-rank off-diagonal blocks), for nrhs column-major vectors.
#include <algorithm>

#include "fifa_apply.cuh"
#include "fifa_common.cuh"
#include "fifa_launch.h"

// ---------------------------------------------------------------------------
// Level sweep, pass 1: partial projections p = Q_side^T v over this CTA's rows
// of one node.  part[cta][(a) * nrhs + j], a < 2cap (a < r: left child rows).
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) k_sweep_proj(const FactDesc* __restrict__ Fd, int lvl, int G,
                                                    const double* __restrict__ v, int nrhs, double* __restrict__ part,
                                                    const int* __restrict__ active) {
  if (active && *active == 0) return;
  const int bi = blockIdx.x / G, g = blockIdx.x % G;
  const int nid = node_id(lvl, bi);
  const int r = Fd->rank[nid];
  if (r == 0) return;
  const int cap = Fd->cap;
  const int64_t n = Fd->n;
  int s, h, e;
  node_range(Fd->bnd, lvl, bi, s, h, e);
  const int len = e - s, rc = (len + G - 1) / G;
  const int r0 = s + min(len, g * rc), r1 = s + min(len, g * rc + rc);
  const T* Qb = (const T*)Fd->Q + (size_t)lvl * cap * n;
  __shared__ double red[40];
  double* out = part + (size_t)blockIdx.x * 2 * cap * SW_RHS_MAX;
  for (int side = 0; side < 2; ++side) {
    const int a0 = side == 0 ? max(r0, s) : max(r0, h);
    const int a1 = side == 0 ? min(r1, h) : min(r1, e);
    for (int a = 0; a < r; ++a) {
      const T* Qc = Qb + (size_t)a * n;
      for (int j = 0; j < nrhs; ++j) {
        const double* vj = v + (size_t)j * n;
        double acc = 0.0;
        for (int p = a0 + threadIdx.x; p < a1; p += blockDim.x) acc += to_d(Qc[p]) * vj[p];
        acc = block_sum(acc, red);
        if (threadIdx.x == 0) out[(side * r + a) * SW_RHS_MAX + j] = acc;
      }
    }
  }
}

// Pass 2: reduce the node's partials (fixed order), t = op(Z) p, v += Q t.
// zsel: 0 -> Zf, 1 -> Zi; ztrans: use the transpose.
template <typename T>
__global__ void __launch_bounds__(256) k_sweep_upd(const FactDesc* __restrict__ Fd, int lvl, int G, double* __restrict__ v,
                                                   int nrhs, const double* __restrict__ part, int zsel, int ztrans,
                                                   const int* __restrict__ active) {
  if (active && *active == 0) return;
  const int bi = blockIdx.x / G, g = blockIdx.x % G, base = blockIdx.x - g;
  const int nid = node_id(lvl, bi);
  const int r = Fd->rank[nid];
  if (r == 0) return;
  const int cap = Fd->cap;
  const int64_t n = Fd->n;
  int s, h, e;
  node_range(Fd->bnd, lvl, bi, s, h, e);
  const int len = e - s, rc = (len + G - 1) / G;
  const int r0 = s + min(len, g * rc), r1 = s + min(len, g * rc + rc);
  const T* Qb = (const T*)Fd->Q + (size_t)lvl * cap * n;
  const int r2 = 2 * r, ld2 = 2 * cap;
  const double* Z = (zsel ? Fd->Zi : Fd->Zf) + (size_t)nid * ld2 * ld2;
  __shared__ double pv[2 * FIFA_CAP_MAX * SW_RHS_MAX];
  __shared__ double tv[2 * FIFA_CAP_MAX * SW_RHS_MAX];
  for (int t = threadIdx.x; t < r2 * nrhs; t += blockDim.x) {
    int a = t / nrhs, j = t % nrhs;
    double acc = 0.0;
    for (int q = 0; q < G; ++q) acc += part[(size_t)(base + q) * 2 * cap * SW_RHS_MAX + a * SW_RHS_MAX + j];
    pv[a * SW_RHS_MAX + j] = acc;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < r2 * nrhs; t += blockDim.x) {
    int a = t / nrhs, j = t % nrhs;
    double acc = 0.0;
    for (int b = 0; b < r2; ++b) acc += (ztrans ? Z[b * ld2 + a] : Z[a * ld2 + b]) * pv[b * SW_RHS_MAX + j];
    tv[a * SW_RHS_MAX + j] = acc;
  }
  __syncthreads();
  for (int p = r0 + threadIdx.x; p < r1; p += blockDim.x) {
    const int off = p < h ? 0 : r;
    double acc[SW_RHS_MAX] = {0.0, 0.0};
    for (int a = 0; a < r; ++a) {
      double q = to_d(Qb[(size_t)a * n + p]);
      for (int j = 0; j < nrhs; ++j) acc[j] += q * tv[(off + a) * SW_RHS_MAX + j];
    }
    for (int j = 0; j < nrhs; ++j) v[(size_t)j * n + p] += acc[j];
  }
}

// Leaf step over all leaves: one warp per leaf.
template <typename T>
__global__ void __launch_bounds__(256) k_sweep_leaf(const FactDesc* __restrict__ Fd, double* __restrict__ v, int nrhs,
                                                    int mode, const int* __restrict__ active) {
  if (active && *active == 0) return;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int L = Fd->L, Bm = Fd->Bm, nleaf = Fd->nleaf;
  if (warp >= nleaf) return;
  const int64_t n = Fd->n;
  const int s = Fd->bnd[bnd_off(L) + warp], e = Fd->bnd[bnd_off(L) + warp + 1];
  const T* Lm = (const T*)Fd->Lleaf + (size_t)warp * Bm * Bm;
  const T* dinv = (const T*)Fd->Ldinv + (size_t)warp * Bm;
  if (nrhs > 1) leaf_warp_apply<T, double, 2>(Lm, dinv, Bm, e - s, v + s, v + n + s, mode, lane);
  else leaf_warp_apply<T, double, 1>(Lm, dinv, Bm, e - s, v + s, nullptr, mode, lane);
}

size_t sweep_fused_smem(int rows, int nrhs, int prec) {
  const size_t esz = prec ? sizeof(float) : sizeof(double);
  return esz * ((size_t)rows * nrhs + 2 * FS_BUF + 256) + 8 +
         (fs_qcap(rows) ? 2 * FS_ZBUF * sizeof(double) + 2 * fs_qcap(rows) * esz : 0) +
         sizeof(unsigned short) * (size_t)rows;
}

template <typename T, int NR, bool BATCH = false>
static int sweep_fused_per_sm(size_t smem) {
  int per_sm = 0;
  ALLOW_SMEM(k_sweep_fused<T, NR, BATCH>);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sweep_fused<T, NR, BATCH>, 256, smem) != cudaSuccess)
    per_sm = 0;
  cudaGetLastError();
  return per_sm;
}

int sweep_fused_coresident(int prec, int rows, int cap) {
  (void)cap;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const size_t smem = sweep_fused_smem(rows, SW_RHS_MAX, prec);
  int optin = 0;
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (smem > (size_t)optin) return 0;
  const int per_sm =
      prec ? std::min(sweep_fused_per_sm<float, 1>(smem), sweep_fused_per_sm<float, 2>(smem))
           : std::min(std::min(sweep_fused_per_sm<double, 1>(smem), sweep_fused_per_sm<double, 2>(smem)),
                      sweep_fused_per_sm<double, 1, true>(smem));
  return sms * per_sm;
}

// nprob FP64 factors of one plan (descriptor array Fd), one right-hand side
// each at vlist[q], in one cooperative launch of 2^ls x nprob CTAs.
cudaError_t launch_sweep_fused_batched(const FactDesc* Fd, int ls, int rows, double* const* vlist, int nprob,
                                       int mode, double* part, unsigned int* bar, int* abort_flag, size_t pstride,
                                       cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1u << ls, nprob);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = sweep_fused_smem(rows, 1, 0);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return launch_sweep_fused_t<double, 1, true, false>(cfg, Fd, nullptr, mode, ls, rows, part, bar, abort_flag, nullptr,
                                                      vlist, pstride);
}

cudaError_t launch_sweep_fused(const FactDesc* Fd, int prec, int ls, int rows, int cap, double* v, int nrhs,
                               int mode, double* part, unsigned int* bar, int* abort_flag, bool cluster,
                               cudaStream_t st, const int* active) {
  (void)cap;
  if (cluster) return launch_sweep_cluster(Fd, prec, ls, rows, v, nrhs, mode, part, st, active);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1u << ls);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = sweep_fused_smem(rows, nrhs, prec);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = mode == 5 ? 0 : 1;  // mode 5's CTAs never wait on each other
  cfg.attrs = attr;
  cfg.numAttrs = 1;
#define FS_GO(T, NR) launch_sweep_fused_t<T, NR, false, false>(cfg, Fd, v, mode, ls, rows, part, bar, abort_flag, active)
  if (prec) return nrhs > 1 ? FS_GO(float, 2) : FS_GO(float, 1);
  return nrhs > 1 ? FS_GO(double, 2) : FS_GO(double, 1);
#undef FS_GO
}

// ---------------------------------------------------------------------------
// Posterior at many new inputs: one CTA per new input x*_j takes its whole
// cross-kernel column c through the sweep W^-1 alone (the fused sweep with the
// root's rows in one CTA's shared memory, so no CTA waits on another), and the
// column never leaves the SM:  mu_j = c . alpha (both nullable),
// var_j = tau2 (1 - |W^-1 c|^2).
// Bound by the FP64 pipe: per row one kernel entry, half a leaf's products and
// three per basis column; two CTAs per SM fill it.  n = 10000 (leaves of 39
// rows), 301 inputs: one two-column sweep of the whole GPU per two inputs, with
// five launches, took 14.5 ms.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256, 2)
    k_predict(const HmatDesc* __restrict__ Hd, const FactDesc* __restrict__ Fd, const double* __restrict__ x,
              const double* __restrict__ xstar, int64_t nstar, const double* __restrict__ alpha, double tau2,
              double* __restrict__ mu, double* __restrict__ var) {
  extern __shared__ __align__(16) unsigned char fs_smem[];
  __shared__ double red[40];
  const int n = (int)Fd->n, L = Fd->L, nleaf = Fd->nleaf;
  double* vs = (double*)fs_smem;
  FsShared<double> sh;
  sh.pj = vs + n;
  sh.tv = sh.pj + FS_BUF;
  sh.red = sh.tv + FS_BUF;
  sh.zb = nullptr;
  sh.qb = nullptr;
  sh.qcap = 0;
  sh.lmap = (unsigned short*)(sh.red + 256);
  for (int q = threadIdx.x; q < nleaf; q += blockDim.x) {
    const int s0 = Fd->bnd[bnd_off(L) + q], e0 = Fd->bnd[bnd_off(L) + q + 1];
    for (int p = s0; p < e0; ++p) sh.lmap[p] = (unsigned short)q;
  }
  const double kc = Hd->kc;
  const int kind = Hd->kind;
  for (int64_t j = blockIdx.x; j < nstar; j += gridDim.x) {
    const double xj = xstar[j];
    double acc = 0.0;
    for (int p = threadIdx.x; p < n; p += blockDim.x) {
      const double c = kern_entry(kind, kc, xj, x[p]);
      vs[p] = c;
      if (mu) acc += c * alpha[p];
    }
    if (mu) {
      acc = block_sum(acc, red);
      if (threadIdx.x == 0) mu[j] = acc;
    }
    __syncthreads();
    fs_leaves<double, 1>(Fd, 0, 0, vs, n, 0, 1);
    for (int l = L - 1; l >= 0; --l) fs_local_level<double, 1>(Fd, l, 0, 0, vs, n, 0, n, 1, 0, sh);
    double q = 0.0;
    for (int p = threadIdx.x; p < n; p += blockDim.x) q += vs[p] * vs[p];
    q = block_sum(q, red);
    if (threadIdx.x == 0) var[j] = tau2 * (1.0 - q);
  }
}

static size_t predict_smem(int64_t n) {
  return sizeof(double) * ((size_t)n + 2 * FS_BUF + 256) + sizeof(unsigned short) * (size_t)n;
}

// Whether k_predict takes n training and nstar new inputs: the column fits one
// SM's shared memory, and there are enough new inputs to make up for one CTA's
// sweep being slower than the whole GPU's (one sweep of n = 10000 by one CTA
// costs about as much as 40 inputs by two-column launches).
bool predict_many(int64_t n, int64_t nstar) {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return predict_smem(n) + 1024 <= (size_t)optin && nstar >= std::max<int64_t>(8, n / 256);
}

cudaError_t launch_predict(const HmatDesc* Hd, const FactDesc* Fd, int64_t n, const double* x, const double* xstar,
                           int64_t nstar, const double* alpha, double tau2, double* mu, double* var, cudaStream_t st) {
  const size_t smem = predict_smem(n);
  const cudaError_t e = ALLOW_SMEM(k_predict);
  if (e != cudaSuccess) return e;
  k_predict<<<(unsigned)std::min<int64_t>(nstar, 1 << 20), 256, smem, st>>>(Hd, Fd, x, xstar, nstar, alpha, tau2, mu, var);
  return cudaGetLastError();
}

size_t mv_fused_smem(int rows) {
  return sizeof(double) * ((size_t)rows * SW_RHS_MAX + MV_PROJ_BUF + MV_THREADS_MAX) + sizeof(int) * (size_t)rows;
}

template <int RPT, bool BATCH>
static int mv_fused_per_sm_v(int rows) {
  const size_t smem = mv_fused_smem(rows);
  int dev = 0, optin = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (smem > (size_t)optin) return 0;
  ALLOW_SMEM(k_mv_fused<RPT, BATCH>);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_mv_fused<RPT, BATCH>, mv_shape(rows).threads, smem) !=
      cudaSuccess)
    per_sm = 0;
  cudaGetLastError();
  return per_sm;
}

// the smaller of the single-problem and the multi-problem instantiations
template <int RPT>
static int mv_fused_per_sm(int rows) {
  return std::min(mv_fused_per_sm_v<RPT, false>(rows), mv_fused_per_sm_v<RPT, true>(rows));
}

int mv_fused_coresident(int rows) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  switch (mv_shape(rows).rpt) {
    case 1: return sms * mv_fused_per_sm<1>(rows);
    case 2: return sms * mv_fused_per_sm<2>(rows);
    case 4: return sms * mv_fused_per_sm<4>(rows);
    case 8: return sms * mv_fused_per_sm<8>(rows);
    case 16: return sms * mv_fused_per_sm<16>(rows);
    default: return 0;
  }
}

// nprob H-matrices of one plan (descriptor array Hd), one right-hand side each
// (xlist[q] -> ylist[q]), in one cooperative launch of 2^ls x nprob CTAs.
cudaError_t launch_mv_fused_batched(const HmatDesc* Hd, int ls, int rows, const double* const* xlist,
                                    double* const* ylist, int nprob, double* part, unsigned int* bar, size_t pstride,
                                    cudaStream_t st) {
#define MVB(R) launch_mv_fused_t<R, true, false>(Hd, ls, rows, nullptr, 1, nullptr, part, bar, st, nullptr, xlist, ylist, nprob, pstride)
  switch (mv_shape(rows).rpt) {
    case 1: return MVB(1);
    case 2: return MVB(2);
    case 4: return MVB(4);
    case 8: return MVB(8);
    case 16: return MVB(16);
    default: return cudaErrorInvalidValue;
  }
#undef MVB
}

cudaError_t launch_mv_fused(const HmatDesc* Hd, int ls, int rows, const double* x, int nrhs, double* y, double* part,
                            unsigned int* bar, bool cluster, cudaStream_t st, const int* active) {
  if (cluster) return launch_mv_cluster(Hd, ls, rows, x, nrhs, y, part, st, active);
  switch (mv_shape(rows).rpt) {
    case 1: return launch_mv_fused_t<1, false, false>(Hd, ls, rows, x, nrhs, y, part, bar, st, active);
    case 2: return launch_mv_fused_t<2, false, false>(Hd, ls, rows, x, nrhs, y, part, bar, st, active);
    case 4: return launch_mv_fused_t<4, false, false>(Hd, ls, rows, x, nrhs, y, part, bar, st, active);
    case 8: return launch_mv_fused_t<8, false, false>(Hd, ls, rows, x, nrhs, y, part, bar, st, active);
    case 16: return launch_mv_fused_t<16, false, false>(Hd, ls, rows, x, nrhs, y, part, bar, st, active);
    default: return cudaErrorInvalidValue;
  }
}

// ---------------------------------------------------------------------------
// H-matrix product y = scale * C~ x + shift * x.
// Pass 1 (one CTA per leaf): per level, the projection of the leaf's rows onto
//   the level's basis: part[(leaf * L + l) * cap + c][j].
// Pass 2 (one CTA per level node side): sum of the partials of its leaves.
//   proj[((l-node) * 2 + side) * cap + c][j].
// Pass 3 (one CTA per leaf): y = scale (D x + sum_l basis_l proj_other) + shift x.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_mv_proj(const HmatDesc* __restrict__ Hd, const double* __restrict__ x, int nrhs,
                                                 double* __restrict__ part, const int* __restrict__ active) {
  if (active && *active == 0) return;
  const int leaf = blockIdx.x;
  const int L = Hd->L, cap = Hd->cap;
  const int64_t n = Hd->n;
  const int* bnd = Hd->bnd;
  const int s = bnd[bnd_off(L) + leaf], e = bnd[bnd_off(L) + leaf + 1], m = e - s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int l = 0; l < L; ++l) {
    const int r = Hd->rank[node_id(l, leaf >> (L - l))];  // level-l ancestor of the leaf
    for (int t = warp; t < r * nrhs; t += nw) {
      const int c = t / nrhs, j = t % nrhs;
      const double* bc = Hd->bases + ((size_t)l * cap + c) * n + s;
      const double* xj = x + (size_t)j * n + s;
      double acc = 0.0;
      for (int i = lane; i < m; i += 32) acc += bc[i] * xj[i];
      acc = warp_sum(acc);
      if (lane == 0) part[(((size_t)leaf * L + l) * cap + c) * SW_RHS_MAX + j] = acc;
    }
  }
}

__global__ void __launch_bounds__(256) k_mv_sum(const HmatDesc* __restrict__ Hd, int nrhs, const double* __restrict__ part,
                                                double* __restrict__ proj, const int* __restrict__ active) {
  if (active && *active == 0) return;
  // blockIdx.x enumerates (level node, side) pairs in heap order: 2 * node + side
  const int L = Hd->L, cap = Hd->cap;
  const int nid = blockIdx.x >> 1, side = blockIdx.x & 1;
  int l = 31 - __clz(nid + 1);
  const int i = nid + 1 - (1 << l);
  const int r = Hd->rank[nid];
  // leaves of this side: child node (l+1, 2i+side) spans 2^(L-l-1) leaves
  const int nl = 1 << (L - l - 1);
  const int first = (2 * i + side) * nl;
  __shared__ double red[40];
  for (int t = 0; t < r * nrhs; ++t) {
    const int c = t / nrhs, j = t % nrhs;
    double acc = 0.0;
    for (int q = threadIdx.x; q < nl; q += blockDim.x)
      acc += part[(((size_t)(first + q) * L + l) * cap + c) * SW_RHS_MAX + j];
    acc = block_sum(acc, red);
    if (threadIdx.x == 0) proj[(((size_t)nid * 2 + side) * cap + c) * SW_RHS_MAX + j] = acc;
  }
}

__global__ void __launch_bounds__(128) k_mv_expand(const HmatDesc* __restrict__ Hd, const double* __restrict__ x, int nrhs,
                                                   const double* __restrict__ proj, double* __restrict__ y,
                                                   const int* __restrict__ active) {
  if (active && *active == 0) return;
  const int leaf = blockIdx.x;
  const int L = Hd->L, cap = Hd->cap, Bm = Hd->Bm;
  const int64_t n = Hd->n;
  const int* bnd = Hd->bnd;
  const double sc = Hd->scale, shf = Hd->shift;
  const int s = bnd[bnd_off(L) + leaf], e = bnd[bnd_off(L) + leaf + 1], m = e - s;
  const double* D = Hd->leaves + (size_t)leaf * Bm * Bm;
  __shared__ double xs[FIFA_LEAF_MAX * SW_RHS_MAX];
  __shared__ double pr[FIFA_LEVELS_MAX * FIFA_CAP_MAX * SW_RHS_MAX];
  __shared__ int rk[FIFA_LEVELS_MAX];
  for (int t = threadIdx.x; t < m * nrhs; t += blockDim.x) {
    int i = t % m, j = t / m;
    xs[j * FIFA_LEAF_MAX + i] = x[(size_t)j * n + s + i];
  }
  for (int l = threadIdx.x; l < L; l += blockDim.x) {
    const int nid = node_id(l, leaf >> (L - l));           // level-l ancestor of the leaf
    rk[l] = Hd->rank[nid];
    const int other = ((leaf >> (L - l - 1)) & 1) ? 0 : 1;  // rows in the left child use V^T x_right
    for (int c = 0; c < rk[l]; ++c)
      for (int j = 0; j < nrhs; ++j)
        pr[(l * FIFA_CAP_MAX + c) * SW_RHS_MAX + j] = proj[(((size_t)nid * 2 + other) * cap + c) * SW_RHS_MAX + j];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    double acc[SW_RHS_MAX] = {0.0, 0.0};
    for (int k = 0; k < m; ++k) {
      double d = D[(size_t)k * Bm + i];
      for (int j = 0; j < nrhs; ++j) acc[j] += d * xs[j * FIFA_LEAF_MAX + k];
    }
    for (int l = 0; l < L; ++l) {
      const double* bl = Hd->bases + (size_t)l * cap * n + s + i;
      for (int c = 0; c < rk[l]; ++c) {
        double b = bl[(size_t)c * n];
        for (int j = 0; j < nrhs; ++j) acc[j] += b * pr[(l * FIFA_CAP_MAX + c) * SW_RHS_MAX + j];
      }
    }
    for (int j = 0; j < nrhs; ++j) {
      double xv = xs[j * FIFA_LEAF_MAX + i];
      const double sh = Hd->diag ? Hd->diag[s + i] : shf;
      y[(size_t)j * n + s + i] = (!Hd->diag && shf == 0.0 && sc == 1.0) ? acc[j] : sc * acc[j] + sh * xv;
    }
  }
}

// ---------------------------------------------------------------------------
cudaError_t launch_sweep_level(const FactDesc* Fd, int prec, int lvl, int nodes, int G, double* v, int nrhs, double* part,
                               int zsel, int ztrans, cudaStream_t st, const int* active) {
  const int grid = nodes * G;
  if (prec) {
    k_sweep_proj<float><<<grid, 256, 0, st>>>(Fd, lvl, G, v, nrhs, part, active);
    k_sweep_upd<float><<<grid, 256, 0, st>>>(Fd, lvl, G, v, nrhs, part, zsel, ztrans, active);
  } else {
    k_sweep_proj<double><<<grid, 256, 0, st>>>(Fd, lvl, G, v, nrhs, part, active);
    k_sweep_upd<double><<<grid, 256, 0, st>>>(Fd, lvl, G, v, nrhs, part, zsel, ztrans, active);
  }
  return cudaGetLastError();
}

cudaError_t launch_sweep_leaf(const FactDesc* Fd, int prec, int nleaf, double* v, int nrhs, int mode, cudaStream_t st,
                              const int* active) {
  const int grid = (nleaf * 32 + 255) / 256;
  if (prec) k_sweep_leaf<float><<<grid, 256, 0, st>>>(Fd, v, nrhs, mode, active);
  else k_sweep_leaf<double><<<grid, 256, 0, st>>>(Fd, v, nrhs, mode, active);
  return cudaGetLastError();
}

cudaError_t launch_matvec(const HmatDesc* Hd, int nleaf, int L, const double* x, int nrhs, double* part, double* proj,
                          double* y, cudaStream_t st, const int* active) {
  if (L > 0) {
    k_mv_proj<<<nleaf, 256, 0, st>>>(Hd, x, nrhs, part, active);
    k_mv_sum<<<2 * ((1 << L) - 1), 256, 0, st>>>(Hd, nrhs, part, proj, active);
  }
  k_mv_expand<<<nleaf, 128, 0, st>>>(Hd, x, nrhs, proj, y, active);
  return cudaGetLastError();
}

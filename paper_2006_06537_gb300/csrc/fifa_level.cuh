// Row tiles, the group reduction and the small Cholesky factor shared by the
// kernels of the factorization (k_node.cu, k_factor.cu).
#pragma once
#include "fifa_common.cuh"

// Reduce `count` doubles of the G partials of this group (slot order fixed)
// into dst; if G == 1 the partial already sits in dst.  The G partials of each
// output are split over the CTA's threads in chunks and the chunk sums
// combined by a pairwise tree in `red` (>= blockDim.x doubles of shared
// memory), so a large group costs a few loads per thread, not G serial ones.
__device__ inline bool group_reduce(double* dst, const double* src_local, int count, int G, int g, int base,
                                    double* part, size_t pstride, unsigned int* bar, unsigned int& phase,
                                    int* status, int* abort_flag, double* red, unsigned int spin) {
  if (G == 1) return true;
  // two slot sets alternate with the barrier count: a slot is rewritten only
  // after a later barrier that every reader of its previous contents has passed
  const size_t set = (size_t)(phase & 1u) * gridDim.x;
  double* mine = part + (set + base + g) * pstride;
  for (int t = threadIdx.x; t < count; t += blockDim.x) mine[t] = src_local[t];
  ++phase;
  if (!group_barrier(bar + base, (unsigned)G * phase, status, abort_flag, spin)) return false;
  const double* slots = part + (set + base) * pstride;
  if (count >= (int)blockDim.x) {
    for (int t = threadIdx.x; t < count; t += blockDim.x) {
      double v = 0.0;
#pragma unroll 8
      for (int q = 0; q < G; ++q) v += __ldcg(slots + (size_t)q * pstride + t);
      dst[t] = v;
    }
    __syncthreads();
    return true;
  }
  const int nch = min(G, (int)blockDim.x / count);
  const int t = threadIdx.x;
  if (t < nch * count) {
    const int o = t % count, ch = t / count;
    double v = 0.0;
#pragma unroll 8
    for (int q = ch; q < G; q += nch) v += __ldcg(slots + (size_t)q * pstride + o);
    red[ch * count + o] = v;
  }
  __syncthreads();
  for (int w = nch; w > 1;) {
    const int hw = (w + 1) / 2;
    for (int i = t; i < (w - hw) * count; i += blockDim.x) red[i] += red[i + hw * count];
    w = hw;
    __syncthreads();
  }
  for (int o = t; o < count; o += blockDim.x) dst[o] = red[o];
  __syncthreads();
  return true;
}

// ---------------------------------------------------------------------------
// Tiled, output-major reductions for the general level kernel: tiles of rows
// are staged in shared memory (coalesced loads, two buffers: the next tile's
// asynchronous copies are in flight while the current one is reduced), each
// output entry is owned by a group of threads that walk disjoint rows of the
// tile, and the groups' partial sums are combined by a short pairwise tree.
// FP64 instructions go to products of nonzero entries only.
// ---------------------------------------------------------------------------
#define LV_TR 128  // rows per staged tile
#define LV_TRP (LV_TR + 1)

__device__ __forceinline__ void pair_decode(int o, int r, int& a, int& b) {
  int rem = o;
  a = 0;
  while (rem >= r - a) {
    rem -= r - a;
    ++a;
  }
  b = a + rem;
}

// 8-byte asynchronous global -> shared copy (cp.async), its group commit and wait.
__device__ __forceinline__ void cp_async8(double* sdst, const void* gsrc) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_prev() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Stage rows [p0, p0 + tr) of ncol columns (column c at col(c)) into a tile
// (column c at c * LV_TRP): asynchronous copies for FP64 storage, converting
// loads for FP32 storage.
template <typename T, typename ColF>
__device__ __forceinline__ void stage_tile(double* tile, int ncol, int p0, int tr, ColF col) {
  for (int i = threadIdx.x; i < ncol * tr; i += blockDim.x) {
    const int c = i / tr, p = i - c * tr;
    const T* src = col(c) + p0 + p;
    if constexpr (sizeof(T) == sizeof(double)) cp_async8(tile + c * LV_TRP + p, src);
    else tile[c * LV_TRP + p] = to_d(*src);
  }
}

// Walk the tiles of rows [a0, a1) with double buffering: body(tile, tr) runs on
// each staged tile by every thread (tbuf: doubles per buffer).
template <typename T, typename ColF, typename BodyF>
__device__ __forceinline__ void tile_walk(double* tile, int tbuf, int ncol, int a0, int a1, ColF col, BodyF body) {
  const int nt = a1 > a0 ? (a1 - a0 + LV_TR - 1) / LV_TR : 0;
  if (nt > 0) stage_tile<T>(tile, ncol, a0, min(LV_TR, a1 - a0), col);
  cp_async_commit();
  for (int k = 0; k < nt; ++k) {
    const int pn = a0 + (k + 1) * LV_TR;
    if (k + 1 < nt) stage_tile<T>(tile + ((k + 1) & 1) * tbuf, ncol, pn, min(LV_TR, a1 - pn), col);
    cp_async_commit();
    cp_async_wait_prev();  // this thread's copies of tile k have landed
    __syncthreads();       // ... and every thread's
    body(tile + (k & 1) * tbuf, min(LV_TR, a1 - (a0 + k * LV_TR)));
    __syncthreads();       // the buffer is free for tile k + 2
  }
}

// 1 / sqrt(d), d > 0: the hardware's approximation y refined by one step of
// Householder's method of third order, y + y e (1/2 + 3/8 e) with e = 1 - d y^2
// (what remains, 5/16 e^3, is below 0.2 u): five FP64 instructions, off by at most
// 1.7 u, u = 2^-53.  Where the approximation would flush a subnormal or d y overflow,
// the library's.  (The library's everywhere takes the same time, but other roundings:
// predictions of an ill-conditioned C~ moved by 2e-9.)
__device__ __forceinline__ double rsqrt_householder(double d) {
  const int ex = (__double2hiint(d) >> 20) & 0x7ff;
  if (ex < 100 || ex > 1900) return rsqrt(d);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  const double e = fma(-(d * y), y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

// One warp, in place: M (r x r symmetric, r <= 16, rows ld apart, upper triangle
// read) = R^T R.  Leaves R above the diagonal of M, its diagonal in Rd, and
// R^-T below and on the diagonal of M (1 / R_kk there).  Left-looking, lane =
// column: row k of R (lanes > k) and of R^-T (lanes < k) are one dot product
// each.  A warp issues an FP64 instruction every 64 cycles (its quarter of the
// SM's FP64 pipe), so what counts is their number, 7 + k for pivot k; the
// diagonal of R is left to one product at the end.  A pivot that is not positive
// is taken as 1 and reported.
static __device__ __noinline__ bool warp_chol_inv(double* M, int ld, int r, double* Rd, int lane) {
  constexpr unsigned FULL = 0xffffffffu;
  bool ok = true;
  double acc = lane < r ? M[lane] : 0.0;  // row 0
  for (int k = 0; k < r; ++k) {
    double d = __shfl_sync(FULL, acc, k);
    const long long bits = __double_as_longlong(d);
    if (!(bits > 0 && bits <= 0x7ff0000000000000LL)) {  // d > 0, tested on the integer pipe
      ok = false;
      d = 1.0;
    }
    const double rs = rsqrt_householder(d);
    const double own = lane == k ? rs : acc * rs;
    if (lane == k) Rd[k] = d;
    if (lane < r) M[k * ld + lane] = own;
    if (k + 1 == r) break;
    // row k + 1 over the rows i <= k: columns of R for lanes > k, of R^-T (from
    // its diagonal on) else
    const bool right = lane > k;
    acc = right && lane < r ? M[(k + 1) * ld + lane] : 0.0;
    acc -= __shfl_sync(FULL, own, k + 1) * own;
    const int lo = right ? 0 : lane;
    const double* col = M + min(lane, r - 1);
    const double* piv = M + k + 1;
    int i = 0;
    for (; i + 4 <= k; i += 4) {
      double a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        a[u] = piv[(i + u) * ld];
        b[u] = i + u >= lo ? col[(i + u) * ld] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) acc -= a[u] * b[u];
    }
    for (; i < k; ++i) acc -= piv[i * ld] * (i >= lo ? col[i * ld] : 0.0);
    __syncwarp();
  }
  __syncwarp();
  if (lane < r) Rd[lane] *= M[lane * ld + lane];  // sqrt(d) = d / sqrt(d)
  __syncwarp();
  return ok;
}

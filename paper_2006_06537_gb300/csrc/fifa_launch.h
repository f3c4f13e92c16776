// Host-side launchers of the device kernels (internal to the library).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <atomic>
#include "fifa_common.cuh"

// Let a kernel take all the dynamic shared memory the device allows, once per
// device: the same value from every thread, so host threads that launch it with
// different sizes never lower each other's limit between its setting and their
// launch.  ALLOW_SMEM(kernel) is a cudaError_t.
inline cudaError_t allow_smem(const void* kernel, std::atomic<unsigned long long>& done) {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
  cudaFuncAttributes a;
  e = cudaFuncGetAttributes(&a, kernel);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)a.sharedSizeBytes);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
  return e;
}
#define ALLOW_SMEM(...)                               \
  ([]() -> cudaError_t {                              \
    static std::atomic<unsigned long long> done{0};   \
    return allow_smem((const void*)(__VA_ARGS__), done); \
  }())

// Assembly launchers take nprob problems of one plan (descriptor arrays,
// blockIdx.y); the grouped ACA's partials / barriers / abort flags of problem q
// sit q * pstride bytes after problem 0's.
cudaError_t launch_leaf_assemble(const HmatDesc* Hd, int nleaf, cudaStream_t st, int nprob = 1);
#define ACA_WARP_MAX 128  // largest side of a block that the warp-per-block ACA takes
// Group sizes of the blocks of levels 0 .. levels - 1 (every block of a level alike).
#define ACA_GROUP_LEVELS 12
struct AcaGroups {
  int levels;
  int G[ACA_GROUP_LEVELS];
};
// ncta CTAs of the grouped blocks (a cooperative launch: they wait on each
// other), by the work list or, with groups, by its group sizes.
cudaError_t launch_aca(const HmatDesc* Hd, const int4* work, int ncta, ArgMax* part, unsigned int* bar, int* abort_flag,
                       cudaStream_t st, int nprob = 1, size_t pstride = 0, const AcaGroups* groups = nullptr);
// one CTA or cluster per block; span: rows and columns of the largest block
cudaError_t launch_aca_blocks(const HmatDesc* Hd, const int4* work, int nsolo, int nwarp, int span, cudaStream_t st,
                              int nprob = 1);
int aca_max_coresident_ctas();

size_t leaf_factor_smem(int Bm, int L, int cap, int prec);
// Doubles per CTA slot of the level kernels' partial sums: the packed Gram
// entries of both sides, r (r + 1) <= cap (cap + 1), and projections of at least
// eight ancestor columns.
__host__ __device__ inline size_t level_part_stride(int cap) { return (size_t)cap * (cap + 1) + (size_t)2 * cap * 8; }
// Nodes of at most this many rows are factored by a thread-block cluster, larger
// ones by a group of CTAs (eight CTAs of a cluster hold 256 rows each, the
// fewest a group's CTA gets).
#define LEVEL_CLUSTER_ROWS 2048
inline bool level_clustered(int side_max) { return 2 * side_max <= LEVEL_CLUSTER_ROWS; }
cudaError_t launch_leaf_factor(const HmatDesc* Hd, const FactDesc* Fd, int prec, int nleaf, int Bm, int L, int cap,
                               cudaStream_t st, int nprob = 1);
#define LEVEL_BUCKETS 3
// Level kernels: rank buckets (.., 4], (4, 16], (16, cap] with groups of G[b]
// CTAs (clusters for small nodes); bucket b uses the barriers at bar + b * bar_stride.
// nprob problems in one launch (grid.y): descriptor arrays, scratch sstride bytes apart.
cudaError_t launch_level(const FactDesc* Fd, int prec, int lvl, int nodes, const int* G, int cap, double* part,
                         unsigned int* bar, int bar_stride, int* abort_flag, int side_max, cudaStream_t st,
                         int nprob = 1, size_t sstride = 0);
// k_node.cu: rank bucket rb (4: all ranks <= 4; 16: ranks in (rlo, 16]) with a
// cluster or a co-resident group of G CTAs per node; ranks <= skip are left out.
cudaError_t launch_node(const FactDesc* Fd, int rb, int rlo, bool cluster, int lvl, int nodes, int G, double* part,
                        unsigned int* bar, int* abort_flag, int skip, cudaStream_t st, int nprob, size_t sstride);
int node_ctas_per_sm(int rb);
int node_cluster_max();  // CTAs of the level kernels' largest cluster on the current device: 16 or 8
// Co-resident CTAs of the level kernel of rank bucket b (0: <= 4, 1: 5..16, 2: > 16).
int level_bucket_coresident(int prec, int b, int cap);
cudaError_t launch_logdet_reduce(const FactDesc* Fd, cudaStream_t st, int nprob = 1);

#define SWEEP_RHS_MAX 2
// active (nullable): when *active == 0 the application / product kernels return at
// once (iterations of a solve that has converged).
cudaError_t launch_sweep_level(const FactDesc* Fd, int prec, int lvl, int nodes, int G, double* v, int nrhs, double* part,
                               int zsel, int ztrans, cudaStream_t st, const int* active = nullptr);
// Fused sweep (one cooperative launch of 2^ls CTAs; rows >= the longest
// level-ls node).  part: 2 ls slots of 2^ls x cap x SWEEP_RHS_MAX doubles; bar,
// zeroed before: the abort flag, then a counter per node of the levels < ls for
// each of two sweeps.  cluster (2^ls <= 8): one cluster instead, which meets at its
// hardware barrier and uses no bar.
#define FS_BAR_COUNTERS 16
inline size_t fs_bar_uints(int ls) { return FS_BAR_COUNTERS + ((size_t)2 << ls); }
#define FS_CTAS_MAX 1024
int sweep_fused_coresident(int prec, int rows, int cap);
// mode 0: W v, 1: W^-1 v, 2: W^T v, 3: W^-T v, 4: W^-T W^-1 v (both inverse sweeps
// in one launch); mode 1 in two launches with the same arithmetic: 5 = its
// leaves and levels >= ls (CTAs independent, launched non-cooperatively; reads
// only those levels of the factor), then 6 = its levels < ls.  Arithmetic in
// the factor's storage precision (prec 1: FP32).
cudaError_t launch_sweep_fused(const FactDesc* Fd, int prec, int ls, int rows, int cap, double* v, int nrhs,
                               int mode, double* part, unsigned int* bar, int* abort_flag, bool cluster,
                               cudaStream_t st, const int* active = nullptr);
// (k_apply_cluster.cu) the same as one cluster of 2^ls <= 8 CTAs
cudaError_t launch_sweep_cluster(const FactDesc* Fd, int prec, int ls, int rows, double* v, int nrhs, int mode,
                                 double* part, cudaStream_t st, const int* active = nullptr);
// nprob FP64 factors of one plan in one launch (one right-hand side each at
// vlist[q]; per-problem partials / barrier / abort flag pstride bytes apart)
cudaError_t launch_sweep_fused_batched(const FactDesc* Fd, int ls, int rows, double* const* vlist, int nprob,
                                       int mode, double* part, unsigned int* bar, int* abort_flag, size_t pstride,
                                       cudaStream_t st);
// Fused H-matrix product (one cooperative launch of 2^ls CTAs, rows <= 4096).
// part: 2^ls * ls * MV_PART_STRIDE doubles; bar, zeroed before: abort flag and counter
// (cluster: not used).
#define MV_FUSED_ROWS_MAX 4096
#define MV_BAR_UINTS 2
int mv_fused_coresident(int rows);
cudaError_t launch_mv_fused(const HmatDesc* Hd, int ls, int rows, const double* x, int nrhs, double* y, double* part,
                            unsigned int* bar, bool cluster, cudaStream_t st, const int* active = nullptr);
// (k_apply_cluster.cu) the same as one cluster of 2^ls <= 8 CTAs, rows <= 1024
cudaError_t launch_mv_cluster(const HmatDesc* Hd, int ls, int rows, const double* x, int nrhs, double* y, double* part,
                              cudaStream_t st, const int* active = nullptr);
// nprob H-matrices of one plan in one launch (one right-hand side each:
// xlist[q] -> ylist[q]; per-problem partials and abort flag / counter pstride
// bytes apart)
cudaError_t launch_mv_fused_batched(const HmatDesc* Hd, int ls, int rows, const double* const* xlist,
                                    double* const* ylist, int nprob, double* part, unsigned int* bar, size_t pstride,
                                    cudaStream_t st);
// Posterior mean (mu, alpha nullable together) and variance at nstar new inputs,
// one CTA each; only where predict_many(n, nstar).
bool predict_many(int64_t n, int64_t nstar);
cudaError_t launch_predict(const HmatDesc* Hd, const FactDesc* Fd, int64_t n, const double* x, const double* xstar,
                           int64_t nstar, const double* alpha, double tau2, double* mu, double* var, cudaStream_t st);
cudaError_t launch_sweep_leaf(const FactDesc* Fd, int prec, int nleaf, double* v, int nrhs, int mode, cudaStream_t st,
                              const int* active = nullptr);
cudaError_t launch_matvec(const HmatDesc* Hd, int nleaf, int L, const double* x, int nrhs, double* part, double* proj,
                          double* y, cudaStream_t st, const int* active = nullptr);

// vector / random / scalar kernels (k_gibbs.cu)
cudaError_t launch_det_exp(const double* in, double* out, int64_t n, cudaStream_t st);
cudaError_t launch_normals(uint64_t seed, uint32_t tag, const uint64_t* iter_dev, uint64_t iter_host, uint64_t stream_id,
                           double* out, int64_t n, cudaStream_t st);
cudaError_t launch_philox(uint64_t seed, const uint32_t* ctr, uint32_t* out, int64_t cnt, cudaStream_t st);
cudaError_t launch_check_sorted(const double* x, int64_t n, int* flag, cudaStream_t st);
// FP64 FMA throughput probe: 16 iters flops per thread, 256 threads per block.
cudaError_t launch_dfma_probe(double* out, int iters, int blocks, cudaStream_t st);

// The fused sweep and the fused H-matrix product as one thread-block cluster: contexts
// with independent CTAs, up to 8192 rows in at most eight CTAs, which the hardware
// schedules together and which meet at its barrier.  Bound by the chain of levels and
// of leaf substitutions on eight SMs.  Against CTAs that polled counters: one W^-1 of
// n = 2048 55 -> 50 us, a product 39 -> 37, a mixed solve 544 -> 513; a solve of
// n = 8192 1133 -> 1098.
#include "fifa_apply.cuh"

static void one_cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int ls) {
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = 1u << ls;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
}

cudaError_t launch_sweep_cluster(const FactDesc* Fd, int prec, int ls, int rows, double* v, int nrhs, int mode,
                                 double* part, cudaStream_t st, const int* active) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3(1u << ls);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = sweep_fused_smem(rows, nrhs, prec);
  cfg.stream = st;
  one_cluster_config(cfg, attr, ls);
#define FS_GO(T, NR) launch_sweep_fused_t<T, NR, false, true>(cfg, Fd, v, mode, ls, rows, part, nullptr, nullptr, active)
  if (prec) return nrhs > 1 ? FS_GO(float, 2) : FS_GO(float, 1);
  return nrhs > 1 ? FS_GO(double, 2) : FS_GO(double, 1);
#undef FS_GO
}

cudaError_t launch_mv_cluster(const HmatDesc* Hd, int ls, int rows, const double* x, int nrhs, double* y, double* part,
                              cudaStream_t st, const int* active) {
#define MV_GO(R) launch_mv_fused_t<R, false, true>(Hd, ls, rows, x, nrhs, y, part, nullptr, st, active)
  switch (mv_shape(rows).rpt) {  // (8192 rows in eight CTAs are 1024 to a CTA)
    case 1: return MV_GO(1);
    case 2: return MV_GO(2);
    case 4: return MV_GO(4);
    default: return cudaErrorInvalidValue;
  }
#undef MV_GO
}

/* The part of the CUDA runtime that k_node.cu calls, for a process with several
 * devices, without a GPU: tests/test_cluster_devices_cpu.py links the compiled
 * k_node.cu against it.  Function attributes belong to the device that was
 * current when they were set, as they do in the runtime; a launch with more than
 * eight CTAs to a cluster is refused unless its function was allowed them on the
 * current device. */
#include <driver_types.h>
#include <stddef.h>
#include <string.h>

#define MAX_DEV 64
#define MAX_FN 64

static int current, nfn, holds16[MAX_DEV], last_cluster;
static const void* fns[MAX_FN];
static int wide[MAX_DEV][MAX_FN];

static int fn_index(const void* f) {
  for (int i = 0; i < nfn; ++i)
    if (fns[i] == f) return i;
  fns[nfn] = f;
  return nfn++;
}

/* the test's controls */
void fake_device(int dev, int can_hold16) {
  current = dev;
  holds16[dev] = can_hold16;
}
int fake_last_cluster(void) { return last_cluster; }

int cudaGetDevice(int* d) {
  *d = current;
  return 0;
}
int cudaGetLastError(void) { return 0; }
int cudaDeviceGetAttribute(int* v, int attr, int dev) {
  (void)attr;
  (void)dev;
  *v = 232448; /* the only one asked for: dynamic shared memory a block may opt in to */
  return 0;
}
int cudaFuncGetAttributes(void* attr, const void* f) {
  (void)f;
  memset(attr, 0, sizeof(struct cudaFuncAttributes));
  return 0;
}
int cudaFuncSetAttribute(const void* f, int attr, int value) {
  if (attr == cudaFuncAttributeNonPortableClusterSizeAllowed) wide[current][fn_index(f)] = value;
  return 0;
}
int cudaOccupancyMaxActiveClusters(int* num, const void* f, const void* cfg) {
  (void)cfg;
  *num = holds16[current] && wide[current][fn_index(f)] ? 1 : 0;
  return 0;
}
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* num, const void* f, int bs, size_t sm, unsigned fl) {
  (void)f;
  (void)bs;
  (void)sm;
  (void)fl;
  *num = 2;
  return 0;
}
int cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  (void)args;
  last_cluster = 0;
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) last_cluster = (int)c->attrs[i].val.clusterDim.x;
  return last_cluster > 8 && !wide[current][fn_index(f)] ? cudaErrorInvalidClusterSize : cudaSuccess;
}

/* what the compiler's host stubs need */
static void* fat;
void** __cudaRegisterFatBinary(void* p) {
  (void)p;
  return &fat;
}
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterFunction(void** h, const char* hf, char* df, const char* n, int t, void* a, void* b, void* c,
                            void* d, int* e) {
  (void)h, (void)hf, (void)df, (void)n, (void)t, (void)a, (void)b, (void)c, (void)d, (void)e;
}
void __cudaRegisterVar(void** h, char* hv, char* da, const char* n, int ext, size_t size, int c, int g) {
  (void)h, (void)hv, (void)da, (void)n, (void)ext, (void)size, (void)c, (void)g;
}
int __cudaGetKernel(void* k, const void* f) {
  (void)k, (void)f;
  return 0;
}
int __cudaLaunchKernel(void* k, ...) {
  (void)k;
  return 0;
}
int __cudaPopCallConfiguration(void* g, ...) {
  (void)g;
  return 0;
}

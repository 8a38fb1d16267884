// The library's host code (csrc/fdlb_api.cpp) on a stand-in for the CUDA runtime
// that keeps "device" memory on the host: what the autotuner adopts, and what
// fdlb_batch_set_tiling makes of the shape it returned.
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "fdlb.h"
#include "fdlb_internal.h"

static int grid_seen = 0, variant_seen = -1;  // of the last stage launched

extern "C" {
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "stand-in"; }
cudaError_t cudaMalloc(void** p, size_t n) { return (*p = std::malloc(n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
// the widest grid of tile shape 1 is the fastest
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = (variant_seen == 1 ? 1.0f : 2.0f) + 1.0f / (float)grid_seen;
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { *e = nullptr; return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
}

namespace fdlb {
bool supported_lattice(int, int, int) { return true; }
int mixed_setup(const DevParams&) { return 0; }
int launch_stage(const DevParams&, int, cudaStream_t) { return 0; }
int launch_init_riemann(const DevParams&, const double*, int, double, double, cudaStream_t) { return 0; }
int launch_moments(const DevParams&, double*, double*, double*, double*, cudaStream_t) { return 0; }
int launch_moments_adjoint(const DevParams&, const double*, const double*, const double*, const double*, double*,
                           cudaStream_t) { return 0; }
int launch_batch_init(const DevParams&, cudaStream_t) { return 0; }
int batch_tile_cells(int variant) { return variant == 1 ? 63 : variant == 2 ? 255 : 127; }
int launch_batch_stage(const DevParams& p, int, cudaStream_t) {
  grid_seen = p.bgrid;
  variant_seen = p.variant;
  return 0;
}
}  // namespace fdlb

static int fails = 0;
#define EXPECT(cond)                                                   \
  do {                                                                 \
    if (!(cond)) {                                                     \
      std::fprintf(stderr, "%s:%d: %s\n", __FILE__, __LINE__, #cond); \
      ++fails;                                                         \
    }                                                                  \
  } while (0)

int main() {
  const int64_t nxs[3] = {256, 1000, 4096};
  const double gms[3] = {1.1, 1.4, 5.0 / 3.0};
  for (int prec : {FDLB_FP64, FDLB_MIXED}) {
    fdlb_ctx* c = nullptr;
    EXPECT(fdlb_create_batch(3, nxs, gms, -0.5, 0.5, 8, 8, 1e-6, 2e-5, prec, nullptr, &c) == FDLB_OK);
    EXPECT(fdlb_step(c, 1) == FDLB_OK);
    const int fresh = grid_seen;
    int variant = -1, ctas = -1;
    EXPECT(fdlb_autotune(c, 1, &variant, &ctas) == FDLB_OK);
    EXPECT(fdlb_step(c, 1) == FDLB_OK);
    const int tuned = grid_seen;
    EXPECT(variant == 1 && variant_seen == 1 && tuned == fresh);
    // another shape, and back to the returned one
    EXPECT(fdlb_batch_set_tiling(c, 0, 4) == FDLB_OK && fdlb_step(c, 1) == FDLB_OK);
    EXPECT(variant_seen == 0 && grid_seen == 4 * 152);
    EXPECT(fdlb_batch_set_tiling(c, variant, ctas) == FDLB_OK && fdlb_step(c, 1) == FDLB_OK);
    EXPECT(variant_seen == variant && grid_seen == tuned);
    // what was accepted and refused stays so
    for (int k : {1, 2, 8, 15, 16, 17, 64}) EXPECT(fdlb_batch_set_tiling(c, 2, k) == FDLB_OK);
    EXPECT(fdlb_batch_set_tiling(c, 2, 0) == FDLB_EINVAL && fdlb_batch_set_tiling(c, 2, 65) == FDLB_EINVAL);
    EXPECT(fdlb_batch_set_tiling(c, 3, 4) == FDLB_EINVAL);
    fdlb_destroy(c);
  }
  if (!fails) std::printf("tiling: ok\n");
  return fails ? 1 : 0;
}

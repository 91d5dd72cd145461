// A CUDA runtime and kernel launchers that only keep a record: linked with the
// library's host code (cat_api.cu, cat_tune.cu) in their place, they show on the
// CPU which launches a call makes, and let a call fail where a test wants it.
//
// fake_log     the launches so far, one per line, and forgets them
// fake_fail    launches named so fail from now on (NULL: none)
// fake_capturing  what cudaStreamIsCapturing returns as its error
// Device memory is host memory; a step on tensor cores takes ten times as long
// as a launch on bit planes (cudaEventElapsedTime).
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <string>

#include "cat_internal.h"

namespace {

std::string g_log, g_fail;
int g_capturing = 0;
float g_clock = 0;

cudaError_t launched(const std::string &what, float ms = 1) {
  if (what == g_fail) return cudaErrorMemoryAllocation;
  g_log += what + "\n";
  g_clock += ms;
  return cudaSuccess;
}

std::string storages(const cat::PlanesGrid &g) {
  const char *name[] = {"u8", "bit1", "nib4"};
  return std::string(name[g.storage_in]) + " to " + name[g.storage_out];
}

CUresult encode_tiled(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                      const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                      CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}

}  // namespace

#define FAKE extern "C" __attribute__((visibility("default")))

FAKE int fake_log(char *out, int size) {
  const int n = (int)g_log.size();
  if (n >= size) return -1;
  memcpy(out, g_log.c_str(), n + 1);
  g_log.clear();
  return n;
}
FAKE void fake_fail(const char *what) { g_fail = what ? what : ""; }
FAKE void fake_capturing(int error) { g_capturing = error; }

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) { return (*p = calloc(1, n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemset(void *p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t) {
  for (size_t y = 0; y < h; ++y) memcpy((char *)d + y * dp, (const char *)s + y * sp, w);
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrComputeCapabilityMajor ? 10 : 3;
  return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) {
  memset(p, 0, sizeof(*p));
  strcpy(p->name, "fake");
  p->multiProcessorCount = 152;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q) {
  *p = (void *)encode_tiled;
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *) {
  a->type = cudaMemoryTypeDevice;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t) new float(0); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete (float *)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { *(float *)e = g_clock; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b) { *ms = *(float *)b - *(float *)a; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
  *s = cudaStreamCaptureStatusNone;
  return (cudaError_t)g_capturing;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { *g = nullptr; return cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *) { return cudaSuccess; }
cudaError_t cudaGraphCreate(cudaGraph_t *g, unsigned) { *g = nullptr; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { *x = (cudaGraphExec_t)1; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return launched("graph"); }
}

namespace cat {
cudaError_t tc_launch(const TcParams &p, int, bool, bool, bool, int, cudaStream_t) {
  return launched("tensor cores", 10.0f * (float)p.n_steps);
}
cudaError_t vn_launch(const TcParams &, int, cudaStream_t) { return launched("tensor cores", 10); }
cudaError_t wide_launch(const TcParams &, int, cudaStream_t) { return launched("tensor cores", 10); }
cudaError_t big_launch(const TcParams &, int, cudaStream_t) { return launched("tensor cores", 10); }
cudaError_t fp4_launch(const TcParams &, int, int, cudaStream_t) { return launched("tensor cores", 10); }
cudaError_t nib_launch(const TcParams &, int, cudaStream_t) { return launched("tensor cores", 10); }
cudaError_t tc_launch_batch(const TcParams &, int, bool, bool, int, cudaStream_t) { return launched("batch tiles", 10); }
cudaError_t mma_launch(const SimpleParams &, int, cudaStream_t) { return launched("fragments", 100); }
cudaError_t stencil_launch(const SimpleParams &, cudaStream_t) { return launched("stencil", 100); }
cudaError_t runsum_launch(const SimpleParams &, cudaStream_t) { return launched("running sums", 100); }
cudaError_t swar_sums_launch(const uint8_t *, int64_t, int64_t, int64_t, const RuleDev &, int32_t *, int64_t,
                             cudaStream_t) {
  return launched("one-bit sums");
}
cudaError_t ghost_fill_launch(uint8_t *, int64_t, int64_t, int64_t, int, bool, cudaStream_t) { return launched("frame"); }
cudaError_t ghost_bits_launch(uint8_t *, int64_t, int64_t, int64_t, cudaStream_t) { return launched("bit frame"); }
cudaError_t pack_bits_launch(const uint8_t *, int64_t, uint8_t *, int64_t, int64_t, int64_t, cudaStream_t) { return cudaSuccess; }
cudaError_t unpack_bits_launch(const uint8_t *, int64_t, uint8_t *, int64_t, int64_t, int64_t, cudaStream_t) { return cudaSuccess; }
cudaError_t pack_nib_launch(const uint8_t *, int64_t, uint8_t *, int64_t, int64_t, int64_t, cudaStream_t) { return cudaSuccess; }
cudaError_t unpack_nib_launch(const uint8_t *, int64_t, uint8_t *, int64_t, int64_t, int64_t, cudaStream_t) { return cudaSuccess; }

// bit planes: preferred wherever they are asked about, one step per launch
bool planes_preferred(const PlanesGrid &g) { return g.rule.nbhd == 0 && g.rule.r <= 16; }
bool planes_steps_preferred(const PlanesGrid &, int64_t) { return true; }
bool planes_few_rows(const PlanesGrid &) { return false; }
cudaError_t swar_step_launch(const PlanesGrid &, cudaStream_t) { return launched("one-bit step"); }
cudaError_t planes_launch(const PlanesGrid &g, cudaStream_t) { return launched("planes " + storages(g)); }
TilePlan planes_tile_plan(const PlanesGrid &, int64_t) { return TilePlan{0, 0}; }
TilePlan planes_tile_steps(const PlanesGrid &, int64_t) { return TilePlan{0, 0}; }
int64_t planes_launches(const PlanesGrid &, int64_t n_steps) { return n_steps; }
TilePlan planes_tile_fixed(const PlanesGrid &, int steps) { return TilePlan{steps, 64}; }
cudaError_t planes_tile_launch(const PlanesGrid &g, const TilePlan &, cudaStream_t) { return launched("tile " + storages(g)); }
cudaError_t planes_prepare(const PlanesGrid &g, const TilePlan &) {
  return "planes " + storages(g) == g_fail ? cudaErrorMemoryAllocation : cudaSuccess;
}
cudaError_t ghost_prepare(int) { return g_fail == "bit frame" ? cudaErrorMemoryAllocation : cudaSuccess; }
struct PlanesBatch {};
cudaError_t planes_batch_create(const std::vector<PlanesBatchItem> &, int, PlanesBatch **out) { *out = new PlanesBatch; return cudaSuccess; }
cudaError_t planes_batch_update(PlanesBatch *, const std::vector<PlanesBatchItem> &) { return cudaSuccess; }
void planes_batch_free(PlanesBatch *b) { delete b; }
cudaError_t planes_batch_add(const PlanesBatch *, int64_t, int, cudaGraph_t) { return launched("batch planes"); }
}  // namespace cat

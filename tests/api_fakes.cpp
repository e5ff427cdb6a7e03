// Fakes of the CUDA runtime for api_harness.cu (which nvcc compiles, and nvcc
// does not let a file define these).  Streams are null and every call has
// finished when it returns.
#include "api_fakes.h"

#include <cstdlib>
#include <cstring>

std::vector<Range> ranges;
std::map<std::string, int> launched;
std::map<std::string, cudaError_t> refused;
static cudaError_t last_error = cudaSuccess;

cudaError_t launch(const char *name) {
  const auto r = refused.find(name);
  if (r != refused.end()) return last_error = r->second;
  ++launched[name];
  return cudaSuccess;
}

static const Range *range_of(const void *p) {
  for (const Range &r : ranges)
    if ((const char *)p >= r.p && (const char *)p < r.p + r.n) return &r;
  return nullptr;
}

extern "C" {
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
  *p = calloc(1, n);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void **d, void *h, unsigned) { *d = h; return cudaSuccess; }
cudaError_t cudaHostGetFlags(unsigned *f, void *p) {
  const Range *r = range_of(p);
  if (!r || r->type != cudaMemoryTypeHost) return last_error = cudaErrorInvalidValue;
  *f = r->flags;
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
  const Range *r = range_of(p);
  a->type = r ? r->type : cudaMemoryTypeUnregistered;
  a->device = 0;
  a->devicePointer = r ? const_cast<void *>(p) : nullptr;
  a->hostPointer = r && r->type == cudaMemoryTypeHost ? const_cast<void *>(p) : nullptr;
  return cudaSuccess;
}
// (a copy to the host refuses a device address)
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  const Range *r = range_of(d);
  if (k == cudaMemcpyDeviceToHost && r && r->type == cudaMemoryTypeDevice)
    return last_error = cudaErrorInvalidValue;
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 1; return cudaSuccess; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = last_error;
  last_error = cudaSuccess;
  return e;
}
const char *cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { *g = nullptr; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) {
  *x = nullptr;
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return launch("graph"); }
// what object files of nvcc register
void **__cudaRegisterFatBinary(void *) {
  static void *handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
}

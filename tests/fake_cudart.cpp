// A CUDA runtime for host-side tests: device memory is host memory, launches do nothing, and a test can make an
// allocation fail or have a kernel report a failure. The library's own objects are linked against it.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

namespace {
long fail_at = 0;    // the fail_at-th allocation from now fails (0: none does)
int reject = 0;      // the check of the line factorisation reports a backward error of this many hundredths
int zero_pivot = 0;  // the dense factorisation reports a zero pivot
int nulls = 0;       // copies, fills and checked launches that were handed a null pointer
int graphs = 0;      // graphs instantiated
int checks = 0;      // line factorisations checked
dim3 conf_grid, conf_block;
size_t conf_smem;
cudaStream_t conf_stream;
std::map<const void *, std::string> &names() {
  static std::map<const void *, std::string> m;
  return m;
}
cudaError_t error = cudaSuccess;
cudaError_t used(const void *p, size_t n) {
  if (p != nullptr || n == 0) return cudaSuccess;
  ++nulls;
  return error = cudaErrorInvalidValue;
}
template <typename T>
T arg(void **args, int i) {
  return *static_cast<T *>(args[i]);
}
cudaError_t launched(const void *f, dim3 g, void **args) {
  if (g.x == 0 || g.y == 0 || g.z == 0 || g.x > 0x7fffffffu || g.y > 65535 || g.z > 65535)
    return error = cudaErrorInvalidConfiguration;
  const std::string &n = names()[f];
  auto has = [&](const char *s) { return n.find(s) != std::string::npos; };
  if (has("line_product_kernel")) used(arg<void *>(args, 0), 1);
  if (has("check_kernel")) {
    ++checks;
    if (arg<double *>(args, 5) != nullptr) *arg<double *>(args, 5) = 0.01 * reject;
  }
  if (has("lu_pivot_kernel")) {  // A, n, k, ipiv, info
    used(arg<void *>(args, 0), 1);
    used(arg<void *>(args, 3), 1);
    if (zero_pivot && arg<int>(args, 2) == 0) *arg<int *>(args, 4) = 1;
  }
  if (has("tri_tile_kernel") || has("permute_kernel")) used(arg<void *>(args, 0), 1);
  if (has("pack_noise_kernel")) {
    used(arg<void *>(args, 0), 1);
    used(arg<void *>(args, 4), 1);
  }
  // norms of one, so that a solve reaches its preconditioner
  if (has("norm2_batch_kernel") && used(arg<void *>(args, 3), 1) == cudaSuccess)
    for (int v = 0; v < 2; ++v) arg<double *>(args, 3)[v] = 1.0;
  return cudaSuccess;
}
}  // namespace

extern "C" {
void fake_fail_at(long n) { fail_at = n; }
void fake_factor(int r, int z) { reject = r, zero_pivot = z; }
int fake_nulls() { return nulls; }
int fake_graphs() { return graphs; }
int fake_checks() { return checks; }

static cudaError_t take(void **p, size_t n) {
  *p = nullptr;
  if (fail_at > 0 && --fail_at == 0) return error = cudaErrorMemoryAllocation;
  *p = std::calloc(n, 1);
  return cudaSuccess;
}
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return take(p, n); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return std::free(p), cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned int) { return take(p, n); }
cudaError_t cudaMallocHost(void **p, size_t n) { return take(p, n); }
cudaError_t cudaFreeHost(void *p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) {
  const cudaError_t e = used(p, n);
  if (e == cudaSuccess) std::memset(p, v, n);
  return e;
}
cudaError_t cudaMemset(void *p, int v, size_t n) { return cudaMemsetAsync(p, v, n, nullptr); }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
  if (used(d, n) != cudaSuccess || used(s, n) != cudaSuccess) return cudaErrorInvalidValue;
  std::memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind k) { return cudaMemcpyAsync(d, s, n, k, nullptr); }

cudaError_t cudaGetLastError() {
  const cudaError_t e = error;
  error = cudaSuccess;
  return e;
}
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t *p, int) { return *p = nullptr, cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned int) {
  return *n = 1, cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *) {
  return *n = 0, cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *) {
  std::memset(a, 0, sizeof(*a));
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) { return *p = nullptr, cudaSuccess; }

cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned int) { return *s = nullptr, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned int) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
  return *s = cudaStreamCaptureStatusNone, cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return *e = nullptr, cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned int) { return *e = nullptr, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { return *ms = 0.f, cudaSuccess; }

cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t *, const cudaGraphEdgeData *,
                                          size_t, cudaStreamCaptureMode) {
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
  return *g = reinterpret_cast<cudaGraph_t>(&graphs), cudaSuccess;
}
cudaError_t cudaGraphCreate(cudaGraph_t *g, unsigned int) {
  return *g = reinterpret_cast<cudaGraph_t>(&graphs), cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) {
  ++graphs;
  return *e = reinterpret_cast<cudaGraphExec_t>(&graphs), cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphGetNodes(cudaGraph_t, cudaGraphNode_t *, size_t *n) { return *n = 0, cudaSuccess; }
cudaError_t cudaGraphNodeGetType(cudaGraphNode_t, cudaGraphNodeType *t) {
  return *t = cudaGraphNodeTypeKernel, cudaSuccess;
}
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle *, cudaGraph_t, unsigned int, unsigned int) {
  return cudaErrorNotSupported;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t *, cudaGraph_t, const cudaGraphNode_t *, const cudaGraphEdgeData *, size_t,
                             cudaGraphNodeParams *) {
  return cudaErrorNotSupported;
}
cudaError_t cudaGraphAddDependencies(cudaGraph_t, const cudaGraphNode_t *, const cudaGraphNode_t *,
                                     const cudaGraphEdgeData *, size_t) {
  return cudaErrorNotSupported;
}

void **__cudaRegisterFatBinary(void *) {
  static void *h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
  names()[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st *s) {
  conf_grid = g, conf_block = b, conf_smem = smem, conf_stream = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) {
  *g = conf_grid, *b = conf_block, *smem = conf_smem, *static_cast<cudaStream_t *>(s) = conf_stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  return *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(f)), cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3, void **args, size_t, cudaStream_t) {
  return launched(k, g, args);
}
cudaError_t cudaLaunchKernel(const void *f, dim3 g, dim3, void **args, size_t, cudaStream_t) {
  return launched(f, g, args);
}
cudaError_t cudaLaunchCooperativeKernel(const void *f, dim3 g, dim3, void **args, size_t, cudaStream_t) {
  return launched(f, g, args);
}
}

// A CUDA runtime without a GPU, for tests of the library's host code: linked with the library's own object
// files in place of the real runtime.  Device memory is host memory (copies and fills above 1 MB are skipped), kernels
// do not run.  What a test needs to see or to cause:
//   * fake_fail_malloc(n): the n-th cudaMalloc from now returns cudaErrorMemoryAllocation (0: none does);
//   * fake_fail_launch(n): the n-th kernel launch from now is refused;
//   * fake_copies_in_flight(): asynchronous copies on streams that have not been waited for since;
//   * fake_unordered_launches(): launches on another stream than the default one that nothing orders after the
//     copies and fills enqueued on the default stream before (cudaMemcpy to the device, cudaMemset);
//   * fake_set_hook(f): every launch calls f(kernel's mangled name, grid, block, arguments), whose result is
//     the kernel's time in microseconds on a modelled device.  Work starts when the host has enqueued it and
//     the device is free; fake_times(h, e): host time per launch, and the device's time between an event and
//     the kernel after it.  Events read the modelled device's clock.
#include <cuda_runtime_api.h>
#include <sys/mman.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

namespace {
std::map<void *, size_t> blocks;  // every live allocation
std::map<const void *, std::string> names;
std::mutex names_lock;
std::map<cudaStream_t, long> copies;  // enqueued since the stream was last waited for
cudaError_t last = cudaSuccess;
long fail_at = 0, fail_launch = 0, unordered = 0;
bool default_pending = false;
double host_now = 0.0, busy_until = 0.0, host_us = 0.0, event_us = 0.0;
double (*hook)(const char *, const unsigned *, const unsigned *, void **) = nullptr;
struct { dim3 grid, block; size_t smem; cudaStream_t s; } conf;
cudaError_t report(cudaError_t e) {
  if (e != cudaSuccess) last = e;
  return e;
}
cudaError_t launch(const void *f, dim3 g, dim3 b, void **args, cudaStream_t s) {
  if (s && default_pending) unordered++;
  const unsigned gg[3] = {g.x, g.y, g.z}, bb[3] = {b.x, b.y, b.z};
  if (fail_launch > 0 && --fail_launch == 0) return report(cudaErrorInvalidConfiguration);
  host_now += host_us;
  const double t = hook ? hook(names[f].c_str(), gg, bb, args) : 0.0;
  busy_until = std::max(busy_until, host_now) + t;
  return cudaSuccess;
}
cudaError_t copy(void *d, const void *s, size_t n) {
  if (n <= (1u << 20)) memcpy(d, s, n);
  return cudaSuccess;
}
int encode_tiled(...) { return 0; }
}  // namespace

extern "C" {

void fake_fail_malloc(long n) { fail_at = n; }
void fake_fail_launch(long n) { fail_launch = n; }
long fake_live_blocks() { return (long)blocks.size(); }
long fake_copies_in_flight() {
  long n = 0;
  for (auto &c : copies) n += c.second;
  return n;
}
long fake_unordered_launches() { return unordered; }
void fake_set_hook(double (*f)(const char *, const unsigned *, const unsigned *, void **)) { hook = f; }
void fake_times(double host, double event) { host_us = host, event_us = event; }

cudaError_t cudaMalloc(void **p, size_t n) {
  *p = nullptr;
  if (fail_at > 0 && --fail_at == 0) return report(cudaErrorMemoryAllocation);
  if (n == 0) return cudaSuccess;
  void *q = mmap(nullptr, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (q == MAP_FAILED) return report(cudaErrorMemoryAllocation);
  blocks[q] = n;
  *p = q;
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
  if (!p) return cudaSuccess;
  auto it = blocks.find(p);
  if (it == blocks.end()) return report(cudaErrorInvalidValue);
  munmap(p, it->second);
  blocks.erase(it);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind k) {
  if (k == cudaMemcpyHostToDevice) default_pending = true;
  return copy(d, s, n);
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st) {
  copies[st]++;
  return copy(d, s, n);
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) {
  if (n <= (1u << 20)) memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) {
  default_pending = true;
  return cudaMemsetAsync(p, v, n, nullptr);
}

cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
const char *cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaGetDevice(int *d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) {
  *v = 152;  // (only the number of SMs is asked for)
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
  *n = 4;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *sym) {
  *p = const_cast<void *>(sym);
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q) {
  *f = (void *)encode_tiled;
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  *s = reinterpret_cast<cudaStream_t>(new char);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  delete reinterpret_cast<char *>(s);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  copies.erase(s);
  if (!s) default_pending = false;
  host_now = std::max(host_now, busy_until);
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) {
  *e = reinterpret_cast<cudaEvent_t>(new double(0.0));
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  delete reinterpret_cast<double *>(e);
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) {
  *reinterpret_cast<double *>(e) = std::max(host_now, busy_until);
  busy_until = *reinterpret_cast<double *>(e) + event_us;
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) {
  host_now = std::max(host_now, busy_until);
  return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b) {
  *ms = (float)((*reinterpret_cast<double *>(b) - *reinterpret_cast<double *>(a)) * 1e-3);
  return cudaSuccess;
}

// graphs are not modelled
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return report(cudaErrorNotSupported); }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) { return report(cudaErrorNotSupported); }
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t, cudaStreamCaptureStatus *st, unsigned long long *id, cudaGraph_t *,
                                     const cudaGraphNode_t **, const cudaGraphEdgeData **, size_t *) {
  *st = cudaStreamCaptureStatusNone;
  if (id) *id = 0;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *, cudaGraph_t, unsigned long long) { return report(cudaErrorNotSupported); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return report(cudaErrorNotSupported); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args) {
  return launch(f, c->gridDim, c->blockDim, args, c->stream);
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
  conf = {g, b, smem, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) {
  *g = conf.grid;
  *b = conf.block;
  *smem = conf.smem;
  *reinterpret_cast<cudaStream_t *>(s) = conf.s;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(f));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void **args, size_t, cudaStream_t s) {
  return launch(reinterpret_cast<const void *>(k), g, b, args, s);
}
void **__cudaRegisterFatBinary(void *) {
  static void *handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
  std::lock_guard<std::mutex> l(names_lock);
  names[host] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}

}  // extern "C"

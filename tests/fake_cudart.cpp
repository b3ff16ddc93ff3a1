// A CUDA runtime that launches nothing: the calls libdibr makes, recorded in order as lines of
// text.  Linked with the library's objects in place of the real runtime (tests/fakecuda.py) it
// runs the host code without a GPU: which launches, copies and waits a call makes, and what the
// host does when one of them fails.  "Device" memory is host memory that nothing reads.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <condition_variable>
#include <map>
#include <mutex>
#include <string>

#include <cuda_runtime.h>

#include "dibr_internal.h"

namespace {
std::mutex mu;
std::condition_variable cv;
std::string text, text_out;
std::map<const void *, std::string> kernels;
std::string fail_call;  // the call to fail, after fail_skip more of it
int fail_skip = 0;
bool capturing = false, busy = false, gate_closed = false, at_gate = false;
int next_handle = 0;

// Records a line; the error the call returns.
cudaError_t note(const char *call, const std::string &line) {
  std::lock_guard<std::mutex> g(mu);
  text += line + "\n";
  if (fail_call == call && fail_skip-- == 0) {
    fail_call.clear();
    text += std::string("failed ") + call + "\n";
    return cudaErrorLaunchOutOfResources;
  }
  return cudaSuccess;
}

std::string num(long long v) { return " " + std::to_string(v); }
std::string id(const void *p) { return num(static_cast<long long>(reinterpret_cast<uintptr_t>(p))); }
template <class H>
cudaError_t handle(H *out) {
  std::lock_guard<std::mutex> g(mu);
  *out = reinterpret_cast<H>(static_cast<uintptr_t>(++next_handle));
  return cudaSuccess;
}
}  // namespace

extern "C" {
// ---- for the tests
const char *fake_take() {  // what was recorded since the last call
  std::lock_guard<std::mutex> g(mu);
  text_out.swap(text);
  text.clear();
  return text_out.c_str();
}
void fake_fail(const char *call, int skip) {
  std::lock_guard<std::mutex> g(mu);
  fail_call = call;
  fail_skip = skip;
}
void fake_state(int capture, int stream_busy) {
  std::lock_guard<std::mutex> g(mu);
  capturing = capture;
  busy = stream_busy;
}
// closed: the next cudaMemsetAsync waits until the gate is open again (holds the serving loop's
// scheduler at a batch's start)
void fake_gate(int closed) {
  std::unique_lock<std::mutex> g(mu);
  gate_closed = closed;
  cv.notify_all();
  if (!closed) at_gate = false;
}
int fake_at_gate() {
  std::lock_guard<std::mutex> g(mu);
  return at_gate;
}

// ---- the runtime
void **__cudaRegisterFatBinary(void *) {
  static void *h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, void *, void *, void *, void *, int *) {
  std::lock_guard<std::mutex> g(mu);
  kernels[host] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t *, const void *) { return cudaErrorUnknown; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t) { return cudaErrorUnknown; }
unsigned __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return 1; }

cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args) {
  std::string name = "?";
  {
    std::lock_guard<std::mutex> g(mu);
    const std::string &n = kernels[f];
    for (const char *k : {"inpaint_rank_kernel", "inpaint_kernel", "band_kernel", "batch_kernel", "xbf_kernel"})
      if (n.find(k) != std::string::npos) {
        name = k;
        break;
      }
  }
  std::string line = "launch " + name + num(c->gridDim.x) + num(c->blockDim.x);
  if (name == "band_kernel") {
    const auto &a = *static_cast<const dibr::BandArgs *>(args[0]);
    line += num(a.W) + num(a.H) + num(a.row0) + num(a.row1) + num(a.overlap) + id(a.in);
  }
  return note("cudaLaunchKernelExC", line);
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) { return *n = 1, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 0, cudaErrorInvalidValue; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) {
  std::memset(p, 0, sizeof(*p));
  p->major = 10;
  p->minor = 3;
  p->multiProcessorCount = 152;
  p->sharedMemPerBlockOptin = 232448;
  p->sharedMemPerMultiprocessor = 233472;
  return cudaSuccess;
}
CUresult fake_is_capturing(CUstream, CUstreamCaptureStatus *s) {
  std::lock_guard<std::mutex> g(mu);
  *s = capturing ? CU_STREAM_CAPTURE_STATUS_ACTIVE : CU_STREAM_CAPTURE_STATUS_NONE;
  return CUDA_SUCCESS;
}
CUresult fake_query(CUstream) {
  std::lock_guard<std::mutex> g(mu);
  if (capturing) text += "query while capturing\n";
  return capturing ? CUDA_ERROR_STREAM_CAPTURE_UNSUPPORTED : busy ? CUDA_ERROR_NOT_READY : CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *name, void **f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult *q) {
  const std::string n = name;
  *f = n == "cuStreamIsCapturing" ? reinterpret_cast<void *>(fake_is_capturing) : n == "cuStreamQuery" ? reinterpret_cast<void *>(fake_query) : nullptr;
  *q = *f ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}
const char *cudaGetErrorString(cudaError_t) { return "a fake error"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaPeekAtLastError() { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *) { return *p = nullptr, cudaErrorUnknown; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return *p = std::calloc(1, n), cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) {
  if (posix_memalign(p, 256, n)) return cudaErrorMemoryAllocation;
  return note("cudaMallocAsync", "alloc" + num(n));
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return std::free(p), cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return handle(s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return note("cudaStreamSynchronize", "sync"); }
cudaError_t cudaStreamIsCapturing(cudaStream_t st, cudaStreamCaptureStatus *s) {
  CUstreamCaptureStatus c;
  fake_is_capturing(st, &c);
  *s = static_cast<cudaStreamCaptureStatus>(c);
  return cudaSuccess;
}
cudaError_t cudaStreamQuery(cudaStream_t st) {
  const CUresult r = fake_query(st);
  return r == CUDA_ERROR_NOT_READY ? cudaErrorNotReady : r == CUDA_SUCCESS ? cudaSuccess : cudaErrorStreamCaptureUnsupported;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { return note("cudaStreamWaitEvent", "wait" + id(s) + id(e)); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return handle(e); }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return handle(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return note("cudaEventRecord", "record" + id(s) + id(e)); }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.f, cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t n, cudaMemcpyKind k, cudaStream_t) {
  return note("cudaMemcpyAsync", "copy" + num(k) + num(n));
}
cudaError_t cudaMemcpy2DAsync(void *, size_t, const void *, size_t, size_t w, size_t h, cudaMemcpyKind k, cudaStream_t) {
  return note("cudaMemcpy2DAsync", "copy2d" + num(k) + num(w) + num(h));
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) {
  {
    std::unique_lock<std::mutex> g(mu);
    if (gate_closed) {
      at_gate = true;
      cv.wait(g, [] { return !gate_closed; });
    }
  }
  return note("cudaMemsetAsync", "memset" + num(v) + num(n));
}
}

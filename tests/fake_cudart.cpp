// A stand-in for the CUDA runtime on host memory, for tests of the library's host code without a GPU: the library's
// objects are linked with this instead of the runtime. Device memory is host memory (zeroed), copies are done, kernels
// do nothing. fake_fail_alloc(k) / fake_fail_new(k): the k-th device allocation / operator new from now on fails, once.
#include <atomic>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <new>

namespace {
std::atomic<long> fail_alloc{0}, fail_new{0}, live{0}, bytes{0};
bool hit(std::atomic<long> &c) { return c.load() > 0 && c.fetch_sub(1) == 1; }
constexpr int kOk = 0, kNoMemory = 2, kUnsupported = 801;
thread_local int last = 0;
int note(int e) { return e == kOk ? e : (last = e); }
int alloc(void **p, size_t n) {
  *p = nullptr;
  if (hit(fail_alloc)) return note(kNoMemory);
  *p = std::calloc(n ? n : 1, 1);
  if (!*p) return note(kNoMemory);
  ++live;
  bytes += (long)n;
  return kOk;
}
int release(void *p) {
  if (p) --live;
  std::free(p);
  return kOk;
}
char handle;  // every stream, event and registered binary
}  // namespace

void *operator new(std::size_t n) {
  if (hit(fail_new)) throw std::bad_alloc();
  if (void *p = std::malloc(n ? n : 1)) return p;
  throw std::bad_alloc();
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, std::size_t) noexcept { std::free(p); }

extern "C" {
void fake_fail_alloc(long k) { fail_alloc = k; }
void fake_fail_new(long k) { fail_new = k; }
long fake_pending() { return (fail_alloc > 0 ? 1 : 0) + (fail_new > 0 ? 1 : 0); }  // a failure not reached yet
long fake_live() { return live; }                                                    // device allocations held
long fake_bytes() { return bytes; }                                                  // of every device allocation so far

void **__cudaRegisterFatBinary(void *) { return reinterpret_cast<void **>(&handle); }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(...) { return 0; }
int __cudaPopCallConfiguration(void *, void *, size_t *, void *) { return kOk; }
int __cudaGetKernel(void **k, const void *) {
  *k = &handle;
  return kOk;
}
int __cudaLaunchKernel(...) { return kOk; }
int cudaLaunchKernelExC(...) { return kOk; }
int cudaLaunchCooperativeKernel(...) { return kOk; }
int cudaFuncSetAttribute(...) { return kOk; }

int cudaMalloc(void **p, size_t n) { return alloc(p, n); }
int cudaMallocAsync(void **p, size_t n, void *) { return alloc(p, n); }
int cudaMallocFromPoolAsync(void **p, size_t n, void *, void *) { return alloc(p, n); }
int cudaFree(void *p) { return release(p); }
int cudaFreeAsync(void *p, void *) { return release(p); }
int cudaMemcpy(void *d, const void *s, size_t n, int) {
  std::memcpy(d, s, n);
  return kOk;
}
int cudaMemcpyAsync(void *d, const void *s, size_t n, int, void *) {
  std::memcpy(d, s, n);
  return kOk;
}
int cudaMemsetAsync(void *d, int v, size_t n, void *) {
  std::memset(d, v, n);
  return kOk;
}
int cudaMemPoolCreate(void **p, const void *) {
  *p = &handle;
  return kOk;
}
int cudaMemPoolSetAttribute(...) { return kOk; }
int cudaMemPoolDestroy(void *) { return kOk; }

int cudaGetDevice(int *d) { return *d = 0; }
int cudaDeviceGetAttribute(int *v, int, int) {
  *v = 152;
  return kOk;
}
int cudaDeviceSynchronize() { return kOk; }
int cudaGetLastError() {
  const int e = last;
  last = kOk;
  return e;
}
const char *cudaGetErrorName(int) { return "fake"; }
const char *cudaGetErrorString(int) { return "fake"; }
int cudaStreamSynchronize(void *) { return kOk; }
int cudaStreamDestroy(void *) { return kOk; }
int cudaEventDestroy(void *) { return kOk; }

// Not reached by the host code under test.
#define FAKE_UNSUPPORTED(name) \
  int name(...) { return note(kUnsupported); }
FAKE_UNSUPPORTED(cudaStreamCreateWithFlags)
FAKE_UNSUPPORTED(cudaStreamWaitEvent)
FAKE_UNSUPPORTED(cudaStreamBeginCapture)
FAKE_UNSUPPORTED(cudaStreamBeginCaptureToGraph)
FAKE_UNSUPPORTED(cudaStreamEndCapture)
FAKE_UNSUPPORTED(cudaStreamGetCaptureInfo)
FAKE_UNSUPPORTED(cudaStreamUpdateCaptureDependencies)
FAKE_UNSUPPORTED(cudaGraphCreate)
FAKE_UNSUPPORTED(cudaGraphDestroy)
FAKE_UNSUPPORTED(cudaGraphInstantiate)
FAKE_UNSUPPORTED(cudaGraphLaunch)
FAKE_UNSUPPORTED(cudaGraphExecDestroy)
FAKE_UNSUPPORTED(cudaGraphAddNode)
FAKE_UNSUPPORTED(cudaGraphConditionalHandleCreate)
FAKE_UNSUPPORTED(cudaEventCreate)
FAKE_UNSUPPORTED(cudaEventCreateWithFlags)
FAKE_UNSUPPORTED(cudaEventRecord)
FAKE_UNSUPPORTED(cudaEventSynchronize)
FAKE_UNSUPPORTED(cudaEventElapsedTime)
FAKE_UNSUPPORTED(cudaOccupancyMaxActiveBlocksPerMultiprocessor)
FAKE_UNSUPPORTED(cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags)
FAKE_UNSUPPORTED(cudaGetSymbolAddress)
}

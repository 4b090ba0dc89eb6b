// Device status word and CUDA error text.
#include <cuda.h>           // types of the driver's calls (no driver symbol is linked)
#include <cuda_runtime.h>
#include <string.h>

#include <atomic>

#include "../../include/rwkvq.h"
#include "host_util.h"

namespace rwkvq {
__device__ int g_device_status = 0;
static thread_local char t_last_error[256] = "";
static std::atomic<unsigned> g_abort_epoch{0};
unsigned abort_epoch() { return g_abort_epoch.load(); }
void set_last_cuda_error(cudaError_t e) {
  strncpy(t_last_error, cudaGetErrorString(e), sizeof(t_last_error) - 1);
  t_last_error[sizeof(t_last_error) - 1] = 0;
}
// Device address of the status word for the current device (kernels in other translation units
// receive it as an argument).
int* device_status_ptr() {
  static SymbolAddress address;
  void* p = nullptr;
  return address((const void*)&g_device_status, &p) == cudaSuccess ? static_cast<int*>(p) : nullptr;
}
unsigned long long context_id() {
  typedef CUresult (*GetIdFn)(CUcontext, unsigned long long*);
  static const GetIdFn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuCtxGetId", &f, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) f = nullptr;
    return reinterpret_cast<GetIdFn>(f);
  }();
  unsigned long long id = 0;
  return fn && fn(nullptr, &id) == CUDA_SUCCESS ? id : 0ull;
}
int current_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return -1;
  return dev;
}
int sm_count() {
  static std::atomic<int> known[kMaxDevices];
  const int dev = current_device();
  if (dev < 0) return 148;
  int sms = known[dev].load(std::memory_order_relaxed);
  if (sms > 0) return sms;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) return 148;
  known[dev].store(sms, std::memory_order_relaxed);
  return sms;
}
void* pinned_results(size_t bytes) {
  constexpr size_t kLeast = 64 << 10, kMost = 1 << 20;
  struct Buffer { void* p; size_t bytes; unsigned long long context; };
  struct Buffers {
    Buffer of[kMaxDevices];
    ~Buffers() {
      cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;      // as below
      bool relaxed = false;
      for (int d = 0; d < kMaxDevices; ++d) {
        if (!of[d].p) continue;
        if (!relaxed && cudaThreadExchangeStreamCaptureMode(&mode) != cudaSuccess) return;
        relaxed = true;
        // a context that has ended took its buffer with it, and the address may be another allocation's by now
        if ((current_device() == d || cudaSetDevice(d) == cudaSuccess) && context_id() == of[d].context) cudaFreeHost(of[d].p);
      }
    }
  };
  static thread_local Buffers buffers;
  const int dev = current_device();
  const unsigned long long id = dev >= 0 ? context_id() : 0ull;
  if (id == 0 || bytes > kMost) return nullptr;
  Buffer& b = buffers.of[dev];
  if (b.p && b.context == id && b.bytes >= bytes) return b.p;
  // another thread may be capturing a graph, in which an allocation has no part
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  if (cudaThreadExchangeStreamCaptureMode(&mode) != cudaSuccess) return nullptr;
  if (b.p && b.context == id) cudaFreeHost(b.p);      // a context that has ended took its buffer with it
  b = Buffer{nullptr, 0, id};
  size_t want = kLeast;
  while (want < bytes) want *= 2;
  void* p = nullptr;
  const cudaError_t e = cudaHostAlloc(&p, want, cudaHostAllocDefault);
  cudaThreadExchangeStreamCaptureMode(&mode);
  if (e != cudaSuccess) { cudaGetLastError(); return nullptr; }
  b.p = p; b.bytes = want;
  return p;
}
}  // namespace rwkvq

extern "C" {
const char* rwkvq_last_cuda_error(void) { return rwkvq::t_last_error; }

rwkvq_status rwkvq_device_status(void* stream) {
  int v = 0, zero = 0;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemcpyFromSymbolAsync(&v, rwkvq::g_device_status, sizeof(int), 0, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyToSymbolAsync(rwkvq::g_device_status, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return rwkvq::cuda_status(e);
  if (v != 0) rwkvq::g_abort_epoch.fetch_add(1);
  return v == 0 ? RWKVQ_OK : (rwkvq_status)v;
}
}

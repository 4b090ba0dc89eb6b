// Host helpers shared by the .cu translation units: descriptor validation, image offsets,
// CUDA error bookkeeping.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "../../include/rwkvq.h"
#include "format.h"

namespace rwkvq {

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline size_t round_up_sz(size_t v, size_t a) { return (v + a - 1) / a * a; }

inline rwkvq_status check_matrix_desc(const rwkvq_desc* d) {
  if (!d) return RWKVQ_EINVAL;
  if (d->oc <= 0 || d->ic <= 0) return RWKVQ_ESHAPE;
  if (d->method == RWKVQ_SQ) {
    if (d->bits != 3 || d->group != 128) return RWKVQ_EUNSUPPORTED;
    if (d->oc % 16 || d->ic % 128) return RWKVQ_ESHAPE;
    if (d->oc_pad != (int)round_up_sz(d->oc, 128) || d->ic_pad != (int)round_up_sz(d->ic, 256)) return RWKVQ_EINVAL;
  } else if (d->method == RWKVQ_VQ) {
    if ((d->bits != 6 && d->bits != 8) || d->vec_dim != 2 || d->tile != 256) return RWKVQ_EUNSUPPORTED;
    if (d->entries != (1 << d->bits)) return RWKVQ_EINVAL;
    if (d->oc % 256 || d->ic % 256) return RWKVQ_ESHAPE;
    if (d->oc_pad != d->oc || d->ic_pad != d->ic) return RWKVQ_EINVAL;
  } else {
    return RWKVQ_EINVAL;
  }
  return RWKVQ_OK;
}

inline rwkvq_status check_vector_desc(const rwkvq_desc* d, int ic) {
  if (!d) return RWKVQ_EINVAL;
  if (d->method != RWKVQ_VQ || d->oc != 1) return RWKVQ_EINVAL;
  if ((d->bits != 6 && d->bits != 8) || d->vec_dim != 2) return RWKVQ_EUNSUPPORTED;
  if (d->entries != (1 << d->bits)) return RWKVQ_EINVAL;
  if (d->ic != ic || ic % 2) return RWKVQ_ESHAPE;
  return RWKVQ_OK;
}

inline size_t matrix_aux_offset(const rwkvq_desc* d) {
  size_t rb = d->method == RWKVQ_SQ ? RWKVQ_SQ_RECORD_BYTES : rwkvq_vq_record_bytes(d->bits);
  return RWKVQ_HEADER_BYTES + (size_t)(d->oc_pad / 128) * (d->ic_pad / 256) * 8 * rb;
}
inline size_t vector_aux_offset(const rwkvq_desc* d) {
  return RWKVQ_HEADER_BYTES + round_up_sz(((size_t)(d->ic / 2) * d->bits + 7) / 8, 16);
}

constexpr int kMaxDevices = 64;
// Ordinal of the current device, -1 if it cannot be asked or is beyond kMaxDevices.
int current_device();
// Multiprocessors of the current device (148 where it cannot be asked); looked up once per device.
int sm_count();

// Number of the calling thread's context; 0 where it has none yet or the driver cannot be asked.  What is set or looked up in a context ends with
// it (cudaDeviceReset), and the device's next context has another number: whatever is kept between calls is kept with this number beside it.
unsigned long long context_id();

// The opt-in to more than 48 KB of dynamic shared memory holds for a kernel as long as the context: it is asked for once (about 1 us of host
// time) and not at every launch.  One object per kernel, `bytes` the same at every call.  `wide`: clusters of more than eight blocks as well.
struct SmemOptIn {
  std::atomic<unsigned long long> context[kMaxDevices];      // in which it was asked for
  const bool wide = false;
  SmemOptIn() = default;
  explicit SmemOptIn(bool wide_clusters) : context{}, wide(wide_clusters) {}
  cudaError_t operator()(const void* fn, int bytes) {
    const int dev = current_device();
    const unsigned long long id = dev >= 0 ? context_id() : 0ull;
    if (id != 0 && context[dev].load(std::memory_order_relaxed) == id) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && wide) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess && id != 0) context[dev].store(id, std::memory_order_relaxed);
    return e;
  }
};

// Device address of a __device__ variable, looked up once per device and context.  One object per variable.
struct SymbolAddress {
  std::mutex mutex;
  void* at[kMaxDevices];
  unsigned long long context[kMaxDevices];
  cudaError_t operator()(const void* symbol, void** out) {
    const int dev = current_device();
    const unsigned long long id = dev >= 0 ? context_id() : 0ull;
    std::lock_guard<std::mutex> lock(mutex);
    if (id != 0 && context[dev] == id) { *out = at[dev]; return cudaSuccess; }
    const cudaError_t e = cudaGetSymbolAddress(out, symbol);
    if (e == cudaSuccess && id != 0) { at[dev] = *out; context[dev] = id; }
    return e;
  }
};

// Page-locked host memory of the calling thread that a kernel writes a call's results to, for calls that wait for their stream before they return:
// a copy of a few kilobytes to pageable memory behind the kernel took as long as a short kernel (256 x 256 tiles of 4096^2 bf16: 58.7 us the call, 49.0 so, four of them in the Python binding).
// A buffer per thread, device and context, up to 1 MB, freed when the thread ends; nullptr where more is asked for or there is none to be had (the
// caller then copies).  Each call's results are read before the thread makes another call, so no two calls meet in it; a call that ends with an error
// first waits for what it has enqueued (cuda_status_behind).
void* pinned_results(size_t bytes);

void set_last_cuda_error(cudaError_t e);
inline rwkvq_status cuda_status(cudaError_t e) {
  if (e == cudaSuccess) return RWKVQ_OK;
  set_last_cuda_error(e);
  return RWKVQ_ECUDA;
}
// The same for a call that has put work on `s`, which may still be writing its results to the thread's page-locked memory.
inline rwkvq_status cuda_status_behind(cudaError_t e, cudaStream_t s) {
  if (e != cudaSuccess) cudaStreamSynchronize(s);
  return cuda_status(e);
}

}  // namespace rwkvq

// liblrvol renders: the launches of lrvol_render, lrvol_render_trace and
// lrvol_render_noalloc (the last with the library's static scratch).  The kernel
// is in render_kernel.cuh.
#include <mutex>

#include "lrvol_internal.h"

namespace lrvol {
namespace {

cudaError_t launch_render_any(const RenderParams &prm, int degree, int field, int storage, bool trace, cudaStream_t s) {
  const int f = field == kFieldShaded ? 3 : (field == LRVOL_FIELD_MAGNITUDE ? 1 : (field == LRVOL_FIELD_COMPONENT ? 2 : 0));
  switch (storage) {
    case LRVOL_STORE_F32: return launch_render_f32(prm, degree, f, trace, s);
    case LRVOL_STORE_F16: return launch_render_f16(prm, degree, f, trace, s);
    case LRVOL_STORE_BF16: return launch_render_bf16(prm, degree, f, trace, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_render(const RenderParams &prm, int degree, int field, int storage, cudaStream_t s) {
  return launch_render_any(prm, degree, field, storage, false, s);
}

// The same kernel template with the trace compiled in, over the pixel list in
// prm.trace_pix (prm.trace_n entries).
cudaError_t launch_render_trace(const RenderParams &prm, int degree, int field, int storage, cudaStream_t s) {
  if (prm.trace_n == 0) return cudaSuccess;
  return launch_render_any(prm, degree, field, storage, true, s);
}

// ----------------------------------------------------------------------------
// Scratch for lrvol_render_noalloc.  The render kernel needs a little global
// memory beyond its inputs and outputs: the kNumCounters statistics slots (the
// kernel adds to the first three) and a status word in a 64-bit slot, 72 bytes
// in all.  lrvol_render takes them from the handle; lrvol_render_noalloc takes
// them from this file-scope array, so that the call itself allocates nothing.
// Every GPU that loads the library holds these 256 bytes until the process
// exits.  Host code must not pass the symbol itself to a kernel (on the host it
// names a stand-in, not device memory): its device address is looked up once
// per device below and cached for the life of the process (a device reset by
// the caller invalidates it).
// ----------------------------------------------------------------------------
}  // namespace lrvol

static __device__ __align__(256) unsigned long long g_render_scratch[lrvol::kStaticScratchWords];

namespace lrvol {

namespace {
constexpr int kMaxDevices = 256;
std::mutex g_scratch_mutex;
unsigned long long *g_scratch_ptr[kMaxDevices] = {};
}  // namespace

// Device address of g_render_scratch on the current device; resolved on the
// first call for that device, with that device current.
cudaError_t static_scratch(unsigned long long **out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  if (!g_scratch_ptr[dev]) {
    void *ptr = nullptr;
    e = cudaGetSymbolAddress(&ptr, g_render_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_ptr[dev] = static_cast<unsigned long long *>(ptr);
  }
  *out = g_scratch_ptr[dev];
  return cudaSuccess;
}

// Same kernel as launch_render, with the counters and the status word in the
// static scratch (cleared on the stream before the launch).
cudaError_t launch_render_static(RenderParams prm, int degree, int field, int storage, cudaStream_t s,
                                 unsigned long long *counters_out) {
  unsigned long long *scratch = nullptr;
  cudaError_t e = static_scratch(&scratch);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(scratch, 0, sizeof(unsigned long long) * kStaticScratchWords, s);
  if (e != cudaSuccess) return e;
  prm.counters = scratch;
  prm.status = reinterpret_cast<uint32_t *>(scratch + kNumCounters);
  if (prm.row_end > prm.row_begin) {   // an empty row band launches nothing, as in lrvol_render
    e = launch_render(prm, degree, field, storage, s);
    if (e != cudaSuccess) return e;
  }
  if (counters_out) {
    // samples, lookups, rays hit, then the status word widened to 64 bits
    e = cudaMemcpyAsync(counters_out, scratch + kCntSamples, sizeof(unsigned long long) * 3,
                        cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(counters_out + 3, scratch + kNumCounters, sizeof(unsigned long long),
                        cudaMemcpyDeviceToDevice, s);
  }
  return e;
}

}  // namespace lrvol


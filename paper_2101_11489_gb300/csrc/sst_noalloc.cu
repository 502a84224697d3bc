// sst_noalloc.cu -- sst_unpack_noalloc: per-event unpacking that allocates no
// memory at all.
//
// Who needs it: code that may not call cudaMalloc once it is running.  A trigger
// or data-acquisition process typically reserves all device memory up front for
// its own caching allocator, so a library allocation can fail or steal from that
// reserve; cudaMalloc / cudaFree also synchronise the device, which stalls every
// other stream of a real-time pipeline; and some callers run where allocation is
// not allowed at all.  sst_unpack keeps its scratch (look-back states, FED offsets,
// work tickets) in the context and grows it on demand, and a context itself is
// created with cudaMalloc.  This entry point needs neither: its scratch lives in
// the fixed array below, which every GPU that loads the library holds until the
// process exits.
#include <mutex>

#include "sst_internal.h"

namespace {

constexpr uint32_t kMaxFeds = SST_NOALLOC_MAX_FEDS;
constexpr int kMaxDevices = 64;

// The launches' shared state (sst::LookState), about 16 KiB.
static __device__ __align__(256) unsigned long long g_scratch[sst::LookState::words_for(1, kMaxFeds)];

std::mutex g_mu;                    // held while a device's address is looked up
sst::Scratch g_state[kMaxDevices];  // per device; look_unpack.words is g_scratch's address there, once known

// Finds g_scratch's address on the current device (on the first call for that device).
cudaError_t find_scratch(sst::LookState& l) {
  std::lock_guard<std::mutex> lock(g_mu);
  if (l.words) return cudaSuccess;
  void* p = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
  if (e != cudaSuccess) return e;
  l.words = static_cast<unsigned long long*>(p);
  l.events = 1;
  l.items = kMaxFeds;
  return cudaSuccess;
}

}  // namespace

extern "C" sst_status sst_unpack_noalloc(const uint8_t* raw, uint64_t raw_bytes, const uint32_t* fed_len,
                                         uint32_t n_feds, const sst_digis* out, void* stream) {
  if (!raw || !fed_len || !out || !out->strip || !out->adc || !out->chan_off || !out->chan_status || !out->status)
    return SST_ERR_INVALID_ARG;
  if (((uintptr_t)raw & 15u) != 0) return SST_ERR_INVALID_ARG;
  if (n_feds == 0) return SST_ERR_INVALID_ARG;
  if (n_feds > kMaxFeds) return SST_ERR_TOO_LARGE;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return SST_ERR_CUDA;
  sst::Scratch& s = g_state[dev];
  if (find_scratch(s.look_unpack) != cudaSuccess) return SST_ERR_CUDA;
  const cudaError_t e = sst::launch_unpack(raw, raw_bytes, fed_len, n_feds, *out, s, sst::default_shape(),
                                           static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? SST_OK : SST_ERR_CUDA;
}

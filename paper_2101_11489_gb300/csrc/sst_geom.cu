// sst_geom.cu -- local positions of clusters (arXiv 2101.11489 section 4: the
// clusters become hits with positions for the track finder).  The detector
// geometry is not available, so every module gets a strip pitch from the caller
// (a synthetic geometry); the local x of a cluster is measured from the module's
// centre, between strips 127 and 128: x = (barycenter - 128) * pitch[det], one
// binary32 subtraction and one binary32 multiplication, both rounded to nearest.
#include <cmath>

#include "sst_internal.h"

namespace {

// x of a cluster; a module id outside the detector has no position
__device__ __forceinline__ float local_x(uint32_t m, float bary, const float* __restrict__ pitch, uint32_t n_modules) {
  return m < n_modules ? __fmul_rn(__fsub_rn(bary, 128.0f), __ldg(pitch + m)) : __int_as_float(0x7fc00000);
}

// Bound by the latency of a cluster's two dependent loads (module, then its pitch), so a
// thread takes four consecutive clusters, their loads in flight together: in 16-byte
// accesses where the three arrays allow it (WIDE), else one by one.  x may be bary.
// 1.2 M clusters: 12.9 -> 8.9 us from DRAM, 3.4 -> 2.5 from L2; 20,000 from L2 1.3 -> 1.4.
template <bool WIDE>
__global__ void __launch_bounds__(256) k_local_x(const uint32_t* det, const float* bary, uint64_t n,
                                                 const float* __restrict__ pitch, uint32_t n_modules, float* x) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x * 4;
  for (uint64_t k = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4; k < n; k += stride) {
    if (WIDE && k + 4 <= n) {
      const uint4 m = *reinterpret_cast<const uint4*>(det + k);
      const float4 c = *reinterpret_cast<const float4*>(bary + k);
      *reinterpret_cast<float4*>(x + k) =
          make_float4(local_x(m.x, c.x, pitch, n_modules), local_x(m.y, c.y, pitch, n_modules),
                      local_x(m.z, c.z, pitch, n_modules), local_x(m.w, c.w, pitch, n_modules));
      continue;
    }
    float v[4];
#pragma unroll
    for (int i = 0; i < 4; i++)
      if (k + i < n) v[i] = local_x(det[k + i], bary[k + i], pitch, n_modules);
#pragma unroll
    for (int i = 0; i < 4; i++)
      if (k + i < n) x[k + i] = v[i];
  }
}

}  // namespace

using namespace sst;

extern "C" {

sst_status sst_pitch_upload(sst_ctx* ctx, const float* pitch) {
  if (!ctx) return SST_ERR_INVALID_ARG;
  if (!pitch) return set_err(ctx, SST_ERR_INVALID_ARG, "sst_pitch_upload: null pitch");
  const uint32_t n = ctx->n_feds * kCh;
  for (uint32_t i = 0; i < n; i++)
    if (!(pitch[i] > 0.f) || !std::isfinite(pitch[i]))
      return set_err(ctx, SST_ERR_INVALID_ARG, "sst_pitch_upload: pitch must be finite and > 0");
  DeviceGuard g(ctx->device);
  cudaError_t e = cudaSuccess;
  if (!ctx->pitch && (e = cudaMalloc(&ctx->pitch, n * sizeof(float)))) return cuda_err(ctx, e, "cudaMalloc pitch");
  if ((e = cudaMemcpy(ctx->pitch, pitch, n * sizeof(float), cudaMemcpyHostToDevice)))
    return cuda_err(ctx, e, "sst_pitch_upload");
  return SST_OK;
}

sst_status sst_local_x(sst_ctx* ctx, const uint32_t* det, const float* barycenter, uint64_t n, float* x,
                       void* stream) {
  if (!ctx) return SST_ERR_INVALID_ARG;
  if (!ctx->pitch) return set_err(ctx, SST_ERR_STATE, "sst_local_x: no pitch uploaded");
  if (n == 0) return SST_OK;
  if (!det || !barycenter || !x) return set_err(ctx, SST_ERR_INVALID_ARG, "sst_local_x: null pointer");
  DeviceGuard g(ctx->device);
  const uint64_t want = (n + 1023) / 1024;
  const uint64_t cap = (uint64_t)(ctx->n_sm > 0 ? ctx->n_sm : 1) * 8;
  const unsigned grid = (unsigned)(want < cap ? want : cap);
  const bool wide = (((uintptr_t)det | (uintptr_t)barycenter | (uintptr_t)x) & 15u) == 0;
  auto* k = wide ? k_local_x<true> : k_local_x<false>;
  k<<<grid, 256, 0, (cudaStream_t)stream>>>(det, barycenter, n, ctx->pitch, ctx->n_feds * kCh, x);
  return cuda_err(ctx, cudaGetLastError(), "sst_local_x");
}

}  // extern "C"

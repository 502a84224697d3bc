// sst_kernels.cu -- sm_103a kernels for unpacking zero-suppressed FED data and
// three-threshold clustering (arXiv 2101.11489, section 2), per event and batched
// (section 3).
//
// Batches (k_stream, sst_stream.cuh): one lane per channel record, the calibration
// entries of one FE unit in shared memory while all events' records of it pass; where
// the events are too few for that, or their records are read in place from host memory,
// each warp reads them from global memory (k_stream_fed).  The FED headers are checked by
// a prologue (k_fed_scan), which hands every FE unit its byte range; the kept clusters are
// staged per FE unit and event and put in order by k_order.  Placing them with a look-back
// over the units before instead would make every warp wait for units that other CTAs take
// at the same time.
//
// Single events and the smallest batches (k_unpack, k_cluster, k_event, sst_event.cuh):
// one CTA per FED, which finds its record, and with a look-back over the FEDs before it
// its place in the output, by itself; one launch per call.
//
// Floating point in the threshold tests and sums uses explicit round-to-nearest
// intrinsics (__fmul_rn, __fadd_rn, __fdiv_rn, __fsqrt_rn): no multiply-add is
// contracted and results equal a sequential binary32 evaluation bit for bit.
//
// Every device wait (the look-back) has an iteration limit; when it runs out the
// event is flagged SST_EV_TIMEOUT and the CTA carries on without the value.
#include <cstddef>
#include <type_traits>
#include <utility>

#include "sst_internal.h"

namespace sst {

namespace {

// ---------------------------------------------------------------- constants

constexpr uint32_t kLbSpinLimit = 1u << 20;         // polls before giving up (about a second)
constexpr uint64_t kBadOff = ~0ull;                // fed_off marker: record outside the event
constexpr int kFedScanThreads = 128;               // FEDs per k_fed_scan CTA
constexpr int kEvTile = 2048;                      // digis on chip of a CTA that clusters a FED
constexpr int kEvTileLarge = 4096;                 // the same while all CTAs fit the GPU at once with it

// ---------------------------------------------------------------- small helpers

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_release(unsigned long long* p, unsigned long long v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Programmatic dependent launch: a kernel launched with programmatic stream
// serialization may start before the kernel ahead of it on the stream has
// finished; pdl_wait() returns once that kernel has completed and its writes are
// visible (at once for a kernel launched the ordinary way).  pdl_release() lets
// the next such kernel be launched before this one ends.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ uint32_t rd16(const uint8_t* p) { return (uint32_t)p[0] | ((uint32_t)p[1] << 8); }
__device__ __forceinline__ uint32_t rd32(const uint8_t* p) {
  return (uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16) | ((uint32_t)p[3] << 24);
}

// Exclusive block-wide scan of one value per thread (blockDim.x <= 1024).
__device__ uint32_t block_excl_scan(uint32_t v, uint32_t* wsum, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  uint32_t x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < nw ? wsum[lane] : 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, w, d);
      if (lane >= d) w += y;
    }
    wsum[lane] = w;
  }
  __syncthreads();
  const uint32_t pre = warp > 0 ? wsum[warp - 1] : 0u;
  *total = wsum[nw - 1];
  __syncthreads();
  return pre + x - v;
}

__device__ __forceinline__ bool bit(const uint32_t* m, int t) { return (m[t >> 5] >> (t & 31)) & 1u; }

// Centroid of a cluster (a6): its middle without charge, else first + 1/2 + moment /
// charge, the moment taken about its first strip; each operation one binary32
// rounding.  A moment of 0 (every one-strip cluster) is kept from the division, whose
// slow path zeros take: half the instructions of the ordering pass.
__device__ __forceinline__ float centroid(uint32_t lo, uint32_t wd, uint32_t q, uint32_t moment) {
  if (q == 0) return __fadd_rn((float)lo, __fmul_rn(0.5f, (float)wd));
  const float f = __fdiv_rn(__uint2float_rn(moment ? moment : 1u), __uint2float_rn(q));
  return __fadd_rn(__fadd_rn((float)lo, 0.5f), moment ? f : 0.f);
}

#include "sst_stream.cuh"
#include "sst_event.cuh"

// ---------------------------------------------------------------- batches of many events

// a1, FED level: checks FED `fed`'s header (record at raw + fo, len bytes;
// fo == kBadOff when the record lies outside its event) and describes its 8 FE
// units for the batched kernel: d[v] = (byte offset of FE unit v in the record,
// its length | FED status << 16 | has data << 24).  A header is valid when the
// magic, FED id, channel and FE-unit counts and fed_bytes match and the padded FE
// lengths add up to the record length; otherwise every channel of the FED gets
// SST_CH_FED_HDR.  An absent FED (len 0) has no data and no error.
__device__ void describe_fed(const uint8_t* __restrict__ raw, uint64_t fo, uint32_t len, uint32_t fed, uint2* d) {
  uint32_t st = 0, data = 0;
  uint32_t fe_len[kFe], start[kFe];
#pragma unroll
  for (int v = 0; v < kFe; v++) fe_len[v] = start[v] = 0;
  if (fo == kBadOff) {
    st = SST_CH_FED_HDR;
  } else if (len > 0 && len < (uint32_t)kHdr) {
    st = SST_CH_FED_HDR;
  } else if (len > 0) {
    const uint8_t* g = raw + fo;
    uint32_t h[8];
    if ((fo & 15u) == 0) {
      const uint4 a = __ldg(reinterpret_cast<const uint4*>(g)), b = __ldg(reinterpret_cast<const uint4*>(g) + 1);
      h[0] = a.x; h[1] = a.y; h[2] = a.z; h[3] = a.w; h[4] = b.x; h[5] = b.y; h[6] = b.z; h[7] = b.w;
    } else {
#pragma unroll
      for (int i = 0; i < 8; i++) h[i] = rd32(g + 4 * i);
    }
    uint32_t body = 0;
#pragma unroll
    for (int v = 0; v < kFe; v++) {
      fe_len[v] = (h[4 + v / 2] >> (16 * (v & 1))) & 0xFFFFu;
      start[v] = kHdr + body;
      body += (fe_len[v] + 7u) & ~7u;
    }
    const uint32_t total = (kHdr + body + 15u) & ~15u;
    const bool ok = h[0] == SST_FED_MAGIC && (h[1] & 0xFFFFu) == fed && ((h[1] >> 16) & 0xFFu) == (uint32_t)kCh &&
                    (h[1] >> 24) == (uint32_t)kFe && h[2] == len && total == len;
    if (ok) data = 1;
    else st = SST_CH_FED_HDR;
  }
#pragma unroll
  for (int v = 0; v < kFe; v++)
    d[v] = make_uint2(data ? start[v] : 0u, (data ? fe_len[v] : 0u) | (st << 16) | (data << 24));
}

// a1, outer level: byte offset of every FED record (exclusive scan of fed_len per
// event, plus the event's start).  A record that would end past its event is
// marked kBadOff; a size mismatch sets SST_EV_SIZE.  `cpe` CTAs per event, CTA c
// taking the event's FEDs [c * blockDim.x, (c + 1) * blockDim.x) and summing the
// lengths of the FEDs before them itself.  Every FED's header is checked and its FE
// units described (describe_fed).  It is also the launch sequence's prologue: the
// event's last CTA writes its status (zero but SST_EV_SIZE), its first clears the
// staging counters (amp_alloc: when given), the very first clears the work tickets.
// Event e's bytes are [event_off[e], event_end[e]) when event_end is given (events that do not follow
// one another, e.g. read in place from host memory), else [event_off[e],
// event_off[e + 1]).
__global__ void k_fed_scan(const uint64_t* __restrict__ event_off, const uint64_t* __restrict__ event_end,
                           const uint32_t* __restrict__ fed_len, uint32_t n_feds, uint32_t cpe,
                           uint64_t* __restrict__ fed_off, sst_event_status* status, uint32_t* ev_alloc,
                           uint32_t* tickets, const uint8_t* __restrict__ raw, uint2* unit_desc, uint32_t* amp_alloc) {
  __shared__ uint32_t wsum[32];
  __shared__ unsigned long long psum[32];
  pdl_release();
  const uint32_t e = blockIdx.x / cpe, c = blockIdx.x % cpe;
  const uint32_t f0 = c * blockDim.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t ev0 = event_off[e], ev1 = event_end ? event_end[e] : event_off[e + 1];
  if (c == 0 && threadIdx.x == 0) {
    ev_alloc[counter_at(e)] = 0;
    if (amp_alloc) amp_alloc[counter_at(e)] = 0;
  }
  if (e == 0 && c == 0 && threadIdx.x < 2) tickets[threadIdx.x] = 0;
  const uint32_t* len_e = fed_len + (size_t)e * n_feds;
  // bytes of the event's FEDs before this CTA's
  unsigned long long part = 0;
  for (uint32_t i = threadIdx.x; i < f0 && i < n_feds; i += blockDim.x) part += len_e[i];
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) part += __shfl_down_sync(0xffffffffu, part, d);
  if (lane == 0) psum[warp] = part;
  __syncthreads();
  uint64_t pre = 0;
  for (int k = 0; k < (int)(blockDim.x >> 5); k++) pre += psum[k];
  const uint32_t f = f0 + threadIdx.x;
  const uint32_t len = f < n_feds ? len_e[f] : 0u;
  uint32_t tot;
  const uint32_t ex = block_excl_scan(len, wsum, &tot);
  if (f < n_feds) {
    const uint64_t o = ev0 + pre + ex;
    const uint64_t fo = (ev1 >= ev0 && o + len <= ev1) ? o : kBadOff;
    fed_off[(size_t)e * n_feds + f] = fo;
    describe_fed(raw, fo, len, f, unit_desc + ((size_t)e * n_feds + f) * kFe);
  }
  if (c == cpe - 1 && threadIdx.x == 0)
    status[e] = sst_event_status{0u, 0u, ev0 + pre + tot != ev1 ? SST_EV_SIZE : 0u, 0u};
}

// One slot's FE unit `u` of FED item (event, FED), as the prologue described it.
__device__ __forceinline__ cs::SlotSrc slot_src(const uint8_t* __restrict__ raw, const uint64_t* __restrict__ fed_off,
                                                const uint2* __restrict__ unit_desc, size_t item, uint32_t u) {
  const uint2 d = unit_desc[item * kFe + u];
  const uint64_t fo = fed_off[item];
  cs::SlotSrc r{raw, 0u, (d.y >> 16) & 255u, ((d.y >> 24) & 1u) != 0u};
  if (r.data && fo != kBadOff) {
    r.src = raw + fo + d.x;
    r.len = d.y & 0xFFFFu;
  }
  return r;
}

// The bytes that a warp takes next (lane s: slot s) on their way to L2, up to 512 a unit.
__device__ __forceinline__ void prefetch_slots(const cs::SlotSrc& src) {
  const int lane = threadIdx.x & 31, s = lane >> 2;
  const uint8_t* g =
      reinterpret_cast<const uint8_t*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(src.src), s)) +
      128 * (lane & 3);
  const uint32_t len = __shfl_sync(0xffffffffu, src.len, s);
  if (128u * (lane & 3) < len) asm volatile("prefetch.global.L2 [%0];" ::"l"(g));
}

// a7: the FE units of a batch of many events.  A CTA of W warps holds the
// calibration entries of C = 3 W / 2 channels (24 KB for W = 8: one FE unit) in
// shared memory and runs the events' records of those channels against them (`chunk`
// events per tile and CTA), up to 4 U at a time per warp.
//
// Bound by instruction issue (about 70% of the slots) and shared-memory latency.  On
// 64 full-detector events (79.5 MB of records, 29.4 M digis) it takes 185 us, 5,460
// warp instructions per 96 channels, and the calibration is read from DRAM once
// (86 MB).  (The kernel before it expanded every digi into a tile and found its run and
// candidate by warp ballots: 351 us, 11,700 instructions, 840 MB of gathers from L2.)
template <bool AMP, int W, int U>
__global__ void __launch_bounds__(W * 32, 32 / W) k_stream(const uint8_t* __restrict__ raw,
                                                           const uint64_t* __restrict__ fed_off, uint32_t n_events,
                                                           uint32_t n_feds, const uint64_t* __restrict__ clu_off,
                                                           uint64_t out_cap, sst_event_status* status, KParams kp,
                                                           uint2* stage, uint32_t* ev_alloc, uint32_t* seg_cnt,
                                                           uint32_t* seg_start, uint32_t* ticket,
                                                           const uint2* __restrict__ unit_desc, uint32_t chunk,
                                                           uint32_t per_warp, uint32_t resident, cs::Amps am) {
  constexpr int C = 3 * W / 2, kParts = kChPerFe / C;  // channels of the tile, tiles per FE unit
  static_assert(!AMP || sizeof(uint2) * C * kStrips + W * sizeof(cs::WarpT<U>) <= cs::kFromLimit, "Walk::from");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint2* tile = reinterpret_cast<uint2*>(smem_raw);
  cs::WarpT<U>* warps = reinterpret_cast<cs::WarpT<U>*>(smem_raw + sizeof(uint2) * C * kStrips);
  __shared__ int2 mul[C];
  __shared__ uint32_t s_next;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  cs::WarpT<U>& w = warps[warp];
  uint4* spill = kp.spill + (size_t)(blockIdx.x * W + warp) * kSpillRecords;
  uint32_t* amp_spill = AMP ? am.spill + (size_t)(blockIdx.x * W + warp) * kAmpSpill : nullptr;
  const uint32_t chunks = (n_events + chunk - 1) / chunk, n_items = n_feds * kFe * kParts * chunks;
  // Items (a tile and a chunk of events): the CTAs that fit the GPU at once (`resident`)
  // start on the item of their own index, while the prologue still runs; all further
  // ones come from the ticket.
  bool first = true, fresh = true;
  cs::SlotSrc src{raw, 0u, 0u, false};
  uint32_t t = blockIdx.x;
  if (t >= resident) {
    pdl_wait();
    first = false;
    if (threadIdx.x == 0) s_next = resident + atomicAdd(ticket, 1u);
    __syncthreads();
    t = s_next;
    __syncthreads();
  }
  while (t < n_items) {
    const uint32_t tl = t / chunks, fu = tl / kParts, part = tl % kParts;  // tile, FE unit of the detector, half of it
    const uint32_t e_first = t % chunks * chunk, e_end = e_first + chunk < n_events ? e_first + chunk : n_events;
    const uint32_t ch0 = fu * kChPerFe + part * C;                         // first channel of the tile
    const uint8_t* g = reinterpret_cast<const uint8_t*>(kp.calq + (size_t)ch0 * kStrips);
    for (uint32_t i = threadIdx.x; i < C * kStrips * sizeof(uint2) / 16; i += W * 32)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                       (uint32_t)__cvta_generic_to_shared(smem_raw + 16 * i)),
                   "l"(g + 16 * i)
                   : "memory");
    int2 m2 = make_int2(0, 0);
    if (threadIdx.x < C) mul[threadIdx.x] = m2 = __ldg(reinterpret_cast<const int2*>(kp.mul) + ch0 + threadIdx.x);
    if (first) pdl_wait();  // the prologue's tickets, offsets, unit descriptors and counts
    first = false;
    if (threadIdx.x == 0) s_next = resident + atomicAdd(ticket, 1u);
    asm volatile("cp.async.wait_all;" ::: "memory");
    const bool any_div = __syncthreads_or(m2.x < 0 || m2.y < 0);
    const uint32_t next = s_next;
    if (next < n_items) {  // the next tile's entries on their way to L2
      const uint8_t* g2 = reinterpret_cast<const uint8_t*>(kp.calq + (size_t)(next / chunks) * C * kStrips);
      for (uint32_t i = threadIdx.x; i < C * kStrips * sizeof(uint2) / 128; i += W * 32)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(g2 + 128 * i));
    }
    const cs::Channels<C, false> chans{tile, mul, ch0};
    for (uint32_t e0 = e_first + warp * per_warp; e0 < e_end; e0 += W * per_warp) {
      const uint32_t n = e_end - e0 < per_warp ? e_end - e0 : per_warp;
      const uint32_t e = e0 + (lane < (int)n ? lane : 0);
      if (fresh && lane < (int)n) src = slot_src(raw, fed_off, unit_desc, (size_t)e * n_feds + fu / kFe, fu % kFe);
      if (lane >= (int)n) src = cs::SlotSrc{raw, 0u, 0u, false};
      // what this warp takes next: the next events of this item, or its share of the next
      const bool same = e0 + W * per_warp < e_end;
      const uint32_t fu2 = same ? fu : next / chunks / kParts;
      const uint32_t e2 = (same ? e0 + W * per_warp : next % chunks * chunk + warp * per_warp) + lane;
      cs::SlotSrc src2{raw, 0u, 0u, false};
      if (lane < (int)per_warp && e2 < n_events && fu2 < n_feds * kFe)
        src2 = slot_src(raw, fed_off, unit_desc, (size_t)e2 * n_feds + fu2 / kFe, fu2 % kFe);
      cs::process_slots<AMP, C>(
          w, (int)n, (int)part * C, src, e, (((size_t)e * n_feds + fu / kFe) * kFe + fu % kFe) * kParts + part, kp,
          clu_off, out_cap, status, stage, ev_alloc, seg_cnt, seg_start, spill, chans, any_div, am, amp_spill,
          [&] { prefetch_slots(src2); });
      src = src2;
      fresh = false;
    }
    if (e_first + warp * per_warp >= e_end) fresh = true;  // nothing was read ahead
    __syncthreads();
    t = next;
  }
  pdl_release();
}

// a7 for batches of fewer events: a warp takes `units` adjacent FE units of one FED of
// one event (units x 12 channels) and reads their calibration entries from global
// memory, digi by digi.  The tile of k_stream would cost more than these gathers (24 KB
// against about 4 KB per FE unit and event), and its warps would each have only a few
// channels.  FED-major order, so that the warps at work read the same FEDs' entries.
// LINK: the records are read in place from host memory; else the bytes of a warp's next
// item are fetched to L2 while it works.
constexpr int kFedWarps = 8;
struct FedWarp {
  cs::WarpT<2> w;
  int2 mul[kCh];  // the units' APV multipliers
};
template <bool AMP, bool LINK>
__global__ void __launch_bounds__(kFedWarps * 32, 3) k_stream_fed(
    const uint8_t* __restrict__ raw, const uint64_t* __restrict__ fed_off, uint32_t n_events, uint32_t n_feds,
    const uint64_t* __restrict__ clu_off, uint64_t out_cap, sst_event_status* status, KParams kp, uint2* stage,
    uint32_t* ev_alloc, uint32_t* seg_cnt, uint32_t* seg_start, uint32_t* ticket, const uint2* __restrict__ unit_desc,
    uint32_t units, cs::Amps am) {
  static_assert(!AMP || kFedWarps * sizeof(FedWarp) <= cs::kFromLimit, "Walk::from");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  FedWarp& w = reinterpret_cast<FedWarp*>(smem_raw)[warp];
  const uint32_t id = blockIdx.x * kFedWarps + warp, n_warps = gridDim.x * kFedWarps;
  uint4* spill = kp.spill + (size_t)id * kSpillRecords;
  uint32_t* amp_spill = AMP ? am.spill + (size_t)id * kAmpSpill : nullptr;
  const uint32_t parts = kFe / units, per_fed = n_events * parts, n_items = n_feds * per_fed;
  pdl_wait();
  auto unit_of = [&](uint32_t t, uint32_t* e, uint32_t* f, uint32_t* u) {
    const uint32_t r = t % per_fed;
    *f = t / per_fed;
    *e = r / parts;
    *u = r % parts * units;
  };
  auto src_of = [&](uint32_t t) {
    uint32_t e, f, u;
    unit_of(t, &e, &f, &u);
    cs::SlotSrc src{raw, 0u, 0u, false};
    if (t < n_items && lane < (int)units) src = slot_src(raw, fed_off, unit_desc, (size_t)e * n_feds + f, u + lane);
    return src;
  };
  uint32_t t = id;
  cs::SlotSrc src = src_of(t);
  while (t < n_items) {
    uint32_t next = 0, e, f, u;
    if (lane == 0) next = n_warps + atomicAdd(ticket, 1u);
    unit_of(t, &e, &f, &u);
    const uint32_t ch0 = f * kCh + u * kChPerFe;
    bool div = false;
    for (uint32_t i = lane; i < units * kChPerFe; i += 32) {
      w.mul[i] = __ldg(reinterpret_cast<const int2*>(kp.mul) + ch0 + i);
      div |= w.mul[i].x < 0 || w.mul[i].y < 0;
    }
    div = __any_sync(0xffffffffu, div);
    next = __shfl_sync(0xffffffffu, next, 0);
    const cs::SlotSrc src2 = src_of(next);
    const cs::Channels<kChPerFe, true, LINK> chans{kp.calq + (size_t)ch0 * kStrips, w.mul, ch0};
    cs::process_slots<AMP, kChPerFe>(w.w, (int)units, 0, src, e,
                                     ((size_t)e * n_feds + f) * kFe + u + (lane < (int)units ? lane : 0), kp, clu_off,
                                     out_cap, status, stage, ev_alloc, seg_cnt, seg_start, spill, chans, div, am,
                                     amp_spill, [&] {
                                       if (!LINK) prefetch_slots(src2);
                                     });
    src = src2;
    t = next;
  }
  pdl_release();
}

// a6, packed output (events back to back): each event's cluster count from its
// segments' counts, one CTA of 1024 threads per event; the CTA that finishes last
// (counted in *done, which the prologue cleared; no CTA waits for another) scans the
// events' counts: pack_off[e] = clusters of the events before e, pack_off[n_events]
// = all clusters.
__global__ void __launch_bounds__(1024) k_clu_scan(const uint32_t* __restrict__ seg_cnt, uint32_t n_segs,
                                                   sst_event_status* status, uint64_t* pack_off, uint32_t* done) {
  __shared__ uint32_t wsum[32];
  __shared__ uint64_t pcarry_s;
  __shared__ bool last_s;
  const uint32_t e = blockIdx.x;
  uint32_t n = 0;
  for (uint32_t i = threadIdx.x; i < n_segs; i += blockDim.x) n += seg_cnt[(size_t)e * n_segs + i];
  n = __reduce_add_sync(0xffffffffu, n);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = n;
  __syncthreads();
  if (threadIdx.x < 32) {
    n = __reduce_add_sync(0xffffffffu, wsum[threadIdx.x]);
    if (threadIdx.x == 0) {
      status[e].n_clusters = n;
      __threadfence();  // this event's count is visible before it is counted as done
      last_s = atomicAdd(done, 1u) == gridDim.x - 1;
      pcarry_s = 0;
    }
  }
  __syncthreads();
  if (!last_s) return;
  __threadfence();
  const uint32_t n_events = gridDim.x;
  for (uint32_t b = 0; b < n_events; b += blockDim.x) {
    const uint32_t i = b + threadIdx.x;
    const uint32_t n = i < n_events ? __ldcg(&status[i].n_clusters) : 0u;
    uint32_t tot;
    const uint32_t ex = block_excl_scan(n, wsum, &tot);
    const uint64_t carry = pcarry_s;
    if (i < n_events) pack_off[i] = carry + ex;
    __syncthreads();
    if (threadIdx.x == 0) pcarry_s = carry + tot;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    pack_off[n_events] = pcarry_s;
    *done = 0;
  }
}

// a6, output of k_stream: orders and copies the staged clusters (cs::staged_cluster's
// 8 bytes, `chans` channels to a segment) in one pass and forms their centroids.  CTA c of event e takes the event's segments [c * SEGS, (c + 1) * SEGS):
// it sums the counts of the event's segments before them (its place in the
// event), scans its own counts in shared memory, notes every output record's
// segment there, and copies its clusters to one contiguous range of the output,
// thread t taking records t, t + 256, ... (four loads in flight per thread,
// coalesced stores; each segment's staged records are contiguous).  For the 4.8 M
// clusters of 64 full-detector events it moves 116 MB; 33 us from a cold L2, half of
// its issue slots busy.  (8 threads to a segment, without the map: 50 us, the stores
// no longer coalesced.)  The event's
// clusters start at clu_off[e] (its slice; 0 without clu_off), or at pack_off[e]
// when pack_off is given (k_clu_scan computed it and the events' counts); the
// event's last CTA otherwise stores its cluster count.
// AMP: the segments' amplitudes are ordered the same way, and each cluster's amp_first
// is its segment's place plus its own within the segment.
template <int SEGS, bool AMP>
__global__ void __launch_bounds__(256) k_order(const uint2* __restrict__ stage, const uint64_t* __restrict__ clu_off,
                                               const uint64_t* __restrict__ pack_off,
                                               const uint32_t* __restrict__ seg_cnt,
                                               const uint32_t* __restrict__ seg_start, uint32_t n_segs, uint32_t cpe,
                                               sst_clusters out, sst_event_status* status, uint32_t chans,
                                               cs::Amps am) {
  static_assert(SEGS <= 256, "one scan entry per thread, a byte per segment");
  constexpr bool kNoted = SEGS > 16;             // few segments: searched for instead (4 steps, no barriers)
  constexpr uint32_t kMap = kNoted ? 4096 : 1;   // output records whose segments are noted at once
  __shared__ uint32_t s_dest[SEGS + 1], s_start[SEGS];
  __shared__ uint8_t s_seg[kMap];
  __shared__ uint32_t wsum[32];
  pdl_wait();  // the staged clusters and counts
  const uint32_t e = blockIdx.x / cpe, c = blockIdx.x % cpe;
  const uint32_t seg0 = c * SEGS;
  const uint32_t nseg = n_segs - seg0 < (uint32_t)SEGS ? n_segs - seg0 : (uint32_t)SEGS;
  const uint32_t* cnt_e = seg_cnt + (size_t)e * n_segs;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t v = tid < (int)nseg ? __ldg(cnt_e + seg0 + tid) : 0u;
  if (tid < SEGS) s_start[tid] = tid < (int)nseg ? __ldg(seg_start + (size_t)e * n_segs + seg0 + tid) : 0u;
  // clusters of the event's segments before this CTA's
  uint32_t part = 0;
  for (uint32_t i = tid; i < seg0; i += blockDim.x) part += __ldg(cnt_e + i);
  part = __reduce_add_sync(0xffffffffu, part);
  if (lane == 0) wsum[warp] = part;
  __syncthreads();
  uint32_t pre = 0;
  for (int k = 0; k < (int)(blockDim.x >> 5); k++) pre += wsum[k];
  __syncthreads();
  // this CTA's segments: exclusive scan of their counts
  uint32_t tot;
  const uint32_t ex = block_excl_scan(v, wsum, &tot);
  if (tid < SEGS) s_dest[tid] = ex;
  if (tid == 0) s_dest[SEGS] = tot;
  const uint64_t off = clu_off ? clu_off[e] : 0;
  const uint2* src = stage + off;
  const uint64_t dst = (pack_off ? pack_off[e] : off) + pre;
  uint32_t* const det = out.det + dst;
  uint16_t* const first = out.first + dst;
  uint16_t* const width = out.width + dst;
  uint32_t* const charge = out.charge + dst;
  float* const bary = out.barycenter + dst;
  // the amplitudes, a warp per segment
  __shared__ uint32_t s_amp[AMP ? SEGS : 1];  // place of the segment's first amplitude, or kNoAmp
  __shared__ uint32_t s_acnt[AMP ? SEGS : 1], s_afrom[AMP ? SEGS : 1];
  if (AMP) {
    const uint32_t* acnt_e = am.seg_cnt + (size_t)e * n_segs;
    uint32_t before = 0, atot, slice, slice_end;
    for (uint32_t i = tid; i < seg0; i += blockDim.x) before += __ldg(acnt_e + i);
    const uint32_t mine = tid < (int)nseg ? __ldg(acnt_e + seg0 + tid) : 0u;
    __syncthreads();
    block_excl_scan(before, wsum, &before);  // the sum
    const uint32_t place = block_excl_scan(mine, wsum, &atot);
    cs::amp_slice(am.off, am.cap, e, &slice, &slice_end);
    if (tid < (int)nseg) {
      const uint32_t from = __ldg(am.seg_start + (size_t)e * n_segs + seg0 + tid);
      s_acnt[tid] = mine;
      s_afrom[tid] = from == kNoAmp ? 0u : from;
      s_amp[tid] = from == kNoAmp ? kNoAmp : slice + before + place;
    }
    __syncthreads();
    // 16 threads to a segment, four bytes of it in flight each
    for (uint32_t g = tid / 16; g < nseg; g += 16) {
      const uint32_t n = s_acnt[g];
      const uint8_t* from = am.bytes + slice + s_afrom[g];
      uint8_t* to = out.amp + s_amp[g];
      for (uint32_t k = tid % 16; k < n; k += 64) {
        uint8_t b[4];
#pragma unroll
        for (int u = 0; u < 4; u++) b[u] = k + 16 * u < n ? __ldg(from + k + 16 * u) : (uint8_t)0;
#pragma unroll
        for (int u = 0; u < 4; u++)
          if (k + 16 * u < n) to[k + 16 * u] = b[u];
      }
    }
  }
  constexpr int kU = 4;  // records per thread in flight
  if (!kNoted) __syncthreads();
  for (uint32_t m0 = 0; m0 < tot; m0 += kNoted ? kMap : tot) {
    const uint32_t m1 = kNoted && m0 + kMap < tot ? m0 + kMap : tot;
    if (kNoted) __syncthreads();
    if (kNoted && tid < SEGS)
      for (uint32_t d = ex > m0 ? ex : m0; d < ex + v && d < m1; d++) s_seg[d - m0] = (uint8_t)tid;
    if (kNoted) __syncthreads();
    for (uint32_t d0 = m0 + tid; d0 < m1; d0 += kU * blockDim.x) {
      uint2 r[kU];
      uint32_t m[kU];  // the segment's first module
      uint32_t af[kU];
#pragma unroll
      for (int u = 0; u < kU; u++) {
        const uint32_t d = d0 + u * blockDim.x;
        if (d < m1) {
          uint32_t sg = 0;
          if (kNoted) {
            sg = s_seg[d - m0];
          } else {
#pragma unroll
            for (int step = SEGS / 2; step > 0; step >>= 1)
              if (s_dest[sg + step] <= d) sg += step;
          }
          const uint32_t at = s_start[sg] + (d - s_dest[sg]);
          r[u] = __ldg(src + at);
          m[u] = (seg0 + sg) * chans;
          if (AMP) af[u] = s_amp[sg] == kNoAmp ? kNoAmp : s_amp[sg] + __ldg(am.first + off + at);
        }
      }
#pragma unroll
      for (int u = 0; u < kU; u++) {
        const uint32_t d = d0 + u * blockDim.x;
        if (d < m1) {
          const uint32_t lo = r[u].x & 255u, wd = ((r[u].x >> 8) & 255u) + 1u, q = r[u].x >> 16;
          det[d] = m[u] + (r[u].y >> 24);
          first[d] = (uint16_t)lo;
          width[d] = (uint16_t)wd;
          charge[d] = q;
          bary[d] = centroid(lo, wd, q, r[u].y & 0xFFFFFFu);
          if (AMP) out.amp_first[dst + d] = af[u];
        }
      }
    }
  }
  if (!pack_off && c == cpe - 1 && tid == 0) status[e].n_clusters = pre + tot;
}

// ---------------------------------------------------------------- one CTA per FED

// a1 + a2 per event: one CTA per FED, its digis written to the digi SoA at the FED's
// offset from the look-back over the FEDs' digi counts.
template <int TILE>
__global__ void __launch_bounds__(ev::kThreads) k_unpack(const uint8_t* __restrict__ raw, uint64_t raw_bytes,
                                                         const uint32_t* __restrict__ fed_len, sst_digis out,
                                                         ev::Shared sh, int lanes) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using S = ev::Shm<TILE, false>;
  S& s = *reinterpret_cast<S*>(smem_raw);
  const int tid = threadIdx.x;
  pdl_release();
  pdl_wait();
  ev::Lengths lens;
  const uint32_t f = ev::take_item(s, sh, [&] { lens.load(fed_len, sh.n_feds); });
  if (f >= sh.n_items) return;
  uint32_t len;
  bool ok, size_ok, timed_out;
  const uint64_t fo = ev::find_fed(s, lens, fed_len, f, sh.n_feds, 0, raw_bytes, &len, &ok, &size_ok);
  const uint8_t* src = ev::stage_record(s, raw + (ok ? fo : 0), len);
  const bool slots = src == s.region && len <= (uint32_t)ev::kFedBuf;
  const uint32_t total = slots ? ev::parse_record<true>(s, src, len, f, ok) : ev::parse_record<false>(s, src, len, f, ok);
  ev::Counts own;
  own.digis = total;
  own.flags = s.scal[ev::kFlags];
  own.bad = s.scal[ev::kBad];
  if (tid == 0) ev::publish(sh, f, own);
  const bool single = total <= (uint32_t)TILE;
  if (single) {  // while the FEDs before this one publish
    if (slots) ev::emit_slots(s, len);
    else ev::emit_channels(s, src, 0, kCh, lanes);
  }
  const ev::Counts before = ev::look_back<false, true>(s, sh, f, 0, f == sh.n_feds - 1 ? 0u : ev::kNoStatus, own, &timed_out);
  const uint64_t base = before.digis;
  const uint64_t cap = out.capacity;
  for (int c = tid; c <= kCh; c += ev::kThreads) {
    if (c == kCh && f != sh.n_feds - 1) continue;
    const uint64_t v = base + s.chan_cnt[c];
    out.chan_off[(size_t)f * kCh + c] = (uint32_t)(v < cap ? v : cap);
    if (c < kCh) out.chan_status[(size_t)f * kCh + c] = s.chan_st[c];
  }
  for (int c0 = 0; c0 < kCh && total > 0;) {
    const int c1 = single ? kCh : ev::chunk_end<TILE>(s, c0);
    const uint32_t n = s.chan_cnt[c1] - s.chan_cnt[c0];
    if (!single) ev::emit_channels(s, src, c0, c1, lanes);
    const uint64_t o = base + s.chan_cnt[c0];
    for (uint32_t i = tid; i < n; i += ev::kThreads)
      if (o + i < cap) {
        const uint32_t t = s.tile[i];
        out.strip[o + i] = f * (uint32_t)kFedStrips + (t & 0xFFFFu);
        out.adc[o + i] = (uint8_t)(t >> 16);
      }
    if (!single) __syncthreads();
    c0 = c1;
  }
  if (tid != 0) return;
  if (timed_out) ev::flag_timeout(sh, 0, out.status);
  if (f == sh.n_feds - 1) {
    const uint64_t all = base + total;
    out.status->n_digi = (uint32_t)(all < cap ? all : cap);
    out.status->n_clusters = 0;
    out.status->n_bad_channels = before.bad + own.bad;
    ev::write_flags(sh, 0,
                    before.flags | own.flags | (size_ok ? 0u : SST_EV_SIZE) | (all > cap ? SST_EV_DIGI_CAPACITY : 0u),
                    out.status);
  }
}

// The CTA's spill area for a FED of several chunks, or null.
__device__ __forceinline__ uint2* fed_spill(const KParams& kp) {
  const size_t have = (size_t)kp.spill_warps * kSpillRecords * 2 / ev::kFedClusters;  // in 8-byte records
  return blockIdx.x < have ? reinterpret_cast<uint2*>(kp.spill) + (size_t)blockIdx.x * ev::kFedClusters : nullptr;
}

// a3 - a6 per event: one CTA per FED over the digi SoA.  TILE: three CTAs to an SM with the
// larger one, four with the smaller.
template <bool AMP, int TILE>
__global__ void __launch_bounds__(ev::kThreads, TILE == kEvTileLarge ? 3 : 4) k_cluster(sst_digis in, KParams kp,
                                                                                       sst_clusters out,
                                                                                       ev::Shared sh) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using S = ev::Shm<TILE, true>;
  S& s = *reinterpret_cast<S*>(smem_raw);
  const int tid = threadIdx.x;
  pdl_release();
  pdl_wait();
  const uint32_t f = ev::take_item(s, sh, [] {});
  if (f >= sh.n_items) return;
  // channel digi ranges from the CSR row pointers, clamped to the input capacity
  // and to 256 digis per channel, so that malformed input cannot leave the tile
  uint32_t cnt = 0;
  if (tid < kCh) {
    uint64_t a = in.chan_off[(size_t)f * kCh + tid], b = in.chan_off[(size_t)f * kCh + tid + 1];
    if (a > in.capacity) a = in.capacity;
    if (b > in.capacity) b = in.capacity;
    const uint32_t n = b > a ? (uint32_t)(b - a) : 0u;
    cnt = n < (uint32_t)kStrips ? n : (uint32_t)kStrips;
    s.chan_pos[tid] = (uint32_t)a;
    s.chan_st[tid] = 0;
  }
  const uint32_t total = ev::prefix_counts(s, cnt);
  bool whole = true;  // the channels' digis follow one another
  if (tid < kCh) {
    s.mul[2 * tid] = __ldg(kp.mul + ((size_t)f * kCh + tid) * 2);
    s.mul[2 * tid + 1] = __ldg(kp.mul + ((size_t)f * kCh + tid) * 2 + 1);
    whole = cnt == 0 || s.chan_pos[tid] == s.chan_pos[0] + s.chan_cnt[tid];
  }
  whole = __syncthreads_and(whole);
  const uint32_t g0 = f * (uint32_t)kFedStrips;
  const uint2* cal0 = kp.calq + g0;
  // the channel whose range holds digi i of the FED
  auto channel_of = [&](uint32_t i) {
    uint32_t c = 0;
    for (uint32_t step = 64; step > 0; step >>= 1)
      if (c + step < (uint32_t)kCh && s.chan_cnt[c + step] <= i) c += step;
    return c;
  };
  auto load = [&](int c0, int c1) {
    const uint32_t base = s.chan_cnt[c0], n = s.chan_cnt[c1] - base;
    constexpr int kU = 4;  // digis in flight per thread
    for (uint32_t i0 = tid; whole && i0 < n; i0 += kU * ev::kThreads) {
      const size_t a = (size_t)s.chan_pos[0] + base;
      uint32_t key[kU], adc[kU];
      uint2 v[kU];
#pragma unroll
      for (int u = 0; u < kU; u++) {
        const uint32_t i = i0 + u * ev::kThreads;
        key[u] = i < n ? __ldg(in.strip + a + i) - g0 : 0xFFFFFFFFu;
        adc[u] = i < n ? __ldg(in.adc + a + i) : 0u;
      }
#pragma unroll
      for (int u = 0; u < kU; u++) {
        const uint32_t i = base + i0 + u * ev::kThreads, c = key[u] >> 8;
        v[u] = make_uint2(ev::kNeverActive, 0u);
        // a digi that does not belong to the channel whose range it is in takes no part: it
        // is an inactive digi there
        if (c < (uint32_t)kCh && i >= s.chan_cnt[c] && i < s.chan_cnt[c + 1]) v[u] = __ldg(cal0 + key[u]);
        else if (i0 + u * ev::kThreads < n) key[u] = channel_of(i) << 8;
      }
#pragma unroll
      for (int u = 0; u < kU; u++)
        if (i0 + u * ev::kThreads < n) ev::classify(s, i0 + u * ev::kThreads, key[u], adc[u], v[u]);
    }
    if (!whole && tid >= c0 && tid < c1)  // ranges cut by the capacity or malformed: channel by channel
      for (uint32_t k = 0; k < s.chan_cnt[tid + 1] - s.chan_cnt[tid]; k++) {
        const size_t a = (size_t)s.chan_pos[tid] + k;
        const uint32_t key = in.strip[a] - g0;
        const bool mine = (key >> 8) == (uint32_t)tid;
        ev::classify(s, s.chan_cnt[tid] - base + k, mine ? key : (uint32_t)tid << 8, in.adc[a],
                     mine ? cal0[key] : make_uint2(ev::kNeverActive, 0u));
      }
    __syncthreads();
  };
  const ev::Out o{0, out.capacity, 0, AMP ? out.amp_capacity : 0};
  bool timed_out = false;
  ev::Counts before;
  uint32_t amps;
  const uint32_t found = ev::cluster_fed<AMP, TILE>(
      s, kp, f, total, load,
      [&](uint32_t n, uint32_t a) {
        ev::Counts own;
        own.clusters = n;
        own.amps = a;
        if (tid == 0) ev::publish(sh, f, own);
        return before = ev::look_back<AMP, false>(s, sh, f, 0, ev::kNoStatus, own, &timed_out);
      },
      o, out, fed_spill(kp), &amps);
  if (tid != 0) return;
  if (timed_out) ev::flag_timeout(sh, 0, in.status);
  if (f == sh.n_feds - 1) {
    const uint64_t all = (uint64_t)before.clusters + found, strips = before.amps + amps;
    in.status->n_clusters = (uint32_t)(all < out.capacity ? all : out.capacity);
    const uint32_t fl = (all > out.capacity ? SST_EV_CLUSTER_CAPACITY : 0u) |
                        (AMP && strips > out.amp_capacity ? SST_EV_AMP_CAPACITY : 0u);
    if (fl) atomicOr(&in.status->flags, fl);  // beside the unpacking's
  }
}

// a7 for few events: every FED of every event unpacked and clustered by one CTA, the
// digis in shared memory.  Event e's clusters go to its slice [clu_off[e], clu_off[e + 1]) of the output or, with pack_off, right
// after those of the events before it (pack_off[e], which its first CTA writes).  TILE:
// three CTAs to an SM with the larger one, five with the smaller, so that 700 FED records
// are one wave (four: 77 FEDs x 9 events 40 us for 28).
template <bool AMP, int TILE>
__global__ void __launch_bounds__(ev::kThreads, TILE == kEvTileLarge ? 3 : 5) k_event(const uint8_t* __restrict__ raw,
                                                        const uint64_t* __restrict__ event_off,
                                                        const uint64_t* __restrict__ event_end,
                                                        const uint32_t* __restrict__ fed_len, uint32_t n_events,
                                                        const uint64_t* __restrict__ clu_off, sst_clusters out,
                                                        sst_event_status* status, KParams kp, uint64_t* pack_off,
                                                        ev::Shared sh) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using S = ev::Shm<TILE, true>;
  S& s = *reinterpret_cast<S*>(smem_raw);
  const int tid = threadIdx.x;
  pdl_release();
  pdl_wait();
  const uint32_t n_feds = sh.n_feds;
  ev::Lengths lens;
  const uint32_t idx = ev::take_item(s, sh, [&] {
    if (n_events == 1) lens.load(fed_len, n_feds);
  });
  if (idx >= sh.n_items) return;
  const uint32_t e = idx / n_feds, f = idx % n_feds;
  const uint32_t* len_e = fed_len + (size_t)e * n_feds;
  if (n_events > 1) lens.load(len_e, n_feds);
  const uint64_t ev0 = event_off[e], ev1 = event_end ? event_end[e] : event_off[e + 1];
  ev::Out o;
  if (pack_off) {
    o.off = 0;
    o.room = out.capacity;
  } else {
    const uint64_t a = clu_off[e], b = clu_off[e + 1] < out.capacity ? clu_off[e + 1] : out.capacity;
    o.off = a < out.capacity ? a : 0;
    o.room = b > a ? b - a : 0;
  }
  if (AMP) {
    uint64_t a = out.amp_off[e], b = out.amp_off[e + 1];
    if (b > out.amp_capacity) b = out.amp_capacity;
    if (a > b) a = b;
    o.a_off = a;
    o.a_room = b - a;
  }
  uint32_t len;
  bool ok, size_ok, timed_out = false;
  uint32_t first = 0;  // pack_off: clusters of the events before
  const uint64_t fo = ev::find_fed(s, lens, len_e, f, n_feds, ev0, ev1, &len, &ok, &size_ok);
  const uint8_t* g = raw + (ok ? fo : 0);
  const uint8_t* src = ev::stage_record(s, g, len);
  const bool slots = src == s.region && len <= (uint32_t)ev::kFedBuf;
  const uint32_t total = slots ? ev::parse_record<true>(s, src, len, f, ok) : ev::parse_record<false>(s, src, len, f, ok);
  if (tid < 2 * kCh) s.mul[tid] = __ldg(kp.mul + (size_t)f * 2 * kCh + tid);
  const uint2* cal0 = kp.calq + (size_t)f * kFedStrips;
  const uint32_t lo = e * n_feds, from = pack_off ? 0u : lo;
  ev::Counts before;
  uint32_t amps;
  const uint32_t found = ev::cluster_fed<AMP, TILE>(
      s, kp, f, total,
      [&](int c0, int c1) {
        // (the calibration entries take the staged record's place: a FED of several
        // chunks is read from global memory again)
        const bool single = total <= (uint32_t)TILE;
        if (slots && single) ev::emit_slots(s, len);
        else ev::emit_channels(s, single ? src : g, c0, c1, ev::lanes_for(c1 - c0));
        ev::classify_tile(s, cal0, s.chan_cnt[c1] - s.chan_cnt[c0]);
      },
      [&](uint32_t n, uint32_t a) {
        ev::Counts own;
        own.clusters = n;
        own.digis = total;
        own.amps = a;
        own.flags = s.scal[ev::kFlags];
        own.bad = s.scal[ev::kBad];
        if (tid == 0) ev::publish(sh, idx, own);
        before = ev::look_back<AMP, true>(s, sh, idx, from, f == n_feds - 1 ? lo : ev::kNoStatus, own, &timed_out);
        // the clusters, digis and amplitudes before the event's first, which `before` includes
        if (pack_off && e > 0 && (AMP || f == n_feds - 1)) {
          bool to;
          const ev::Counts start = ev::look_back<AMP, false>(s, sh, lo, 0, ev::kNoStatus, ev::Counts{}, &to);
          before.digis -= start.digis;
          before.amps -= start.amps;
          first = start.clusters;
          timed_out |= to;
        }
        return before;
      },
      o, out, fed_spill(kp), &amps);
  if (tid != 0) return;
  if (timed_out) ev::flag_timeout(sh, e, status + e);
  auto place = [&](uint64_t n) { return n < o.room ? n : o.room; };  // clusters stored of n
  if (pack_off && f == 0) pack_off[e] = place(before.clusters);
  if (pack_off && idx + 1 == sh.n_items) pack_off[n_events] = place((uint64_t)before.clusters + found);
  if (f == n_feds - 1) {
    const uint64_t all = (uint64_t)before.clusters + found;
    sst_event_status* st = status + e;
    st->n_digi = (uint32_t)(before.digis + total);
    st->n_clusters = (uint32_t)(place(all) - place(first));
    st->n_bad_channels = before.bad + s.scal[ev::kBad];
    ev::write_flags(sh, e,
                    before.flags | s.scal[ev::kFlags] | (size_ok ? 0u : SST_EV_SIZE) | (all > o.room ? SST_EV_CLUSTER_CAPACITY : 0u) |
                        (AMP && before.amps + amps > o.a_room ? SST_EV_AMP_CAPACITY : 0u),
                    st);
  }
}

// Host batches with amplitudes: the chunk's amp_first values index the chunk's
// amplitude arena; adding the chunk's first byte in the caller's array makes them
// absolute.  The first *count records are rebased (kNoAmp stays).
__global__ void k_rebase_amp(uint32_t* __restrict__ amp_first, const uint64_t* __restrict__ count, uint32_t base) {
  const uint64_t n = *count;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t a = amp_first[i];
    if (a != kNoAmp) amp_first[i] = a + base;
  }
}

__global__ void k_badmask(const uint8_t* __restrict__ bad, uint32_t* __restrict__ mask, uint64_t n_words) {
  const uint64_t w = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= n_words) return;
  uint32_t m = 0;
  for (int b = 0; b < 32; b++) m |= (bad[w * 32 + b] != 0 ? 1u : 0u) << b;
  mask[w] = m;
}

// Per APV, the charge multiplier of the clusterizers: M with (adc * M + 2^21) >> 22
// equal, for every ADC 1..253, to the ADC divided by the APV's gain, rounded half
// up and capped at 254, each operation one binary32 rounding (section 2: charge
// corrected by the strip's gain); checked here for all of them.  Of U[0.8, 1.2]
// gains all but 5 in 100,000 have one within 4 of 2^22 / gain (a quotient that
// rounds up to a half has none); for those, and for gains below 1/4, where the
// product would pass 32 bits, the bits of -gain: the kernels then divide, and the
// streams take walk_any for the FE unit's channels (16 events with amplitudes and one such
// APV in 1,000: 180 us for 175; all gains below 1/4: 148, of which the division is 2).
__global__ void k_gain_pack(const float* __restrict__ gain, int32_t* __restrict__ mul, uint32_t n_apv) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_apv) return;
  const float g = gain[i];
  int32_t found = __float_as_int(-g);
  if (g >= 0.2500005f) {
    const int32_t m0 = __float2int_rn(__fdiv_rn((float)(1u << kMulShift), g));
    for (int k = 0; k < 9 && found < 0; k++) {
      const int32_t m = m0 + ((k & 1) ? (k + 1) / 2 : -(k / 2));
      if (m < 0) continue;
      bool ok = true;
      for (uint32_t a = 1; a < 254u && ok; a++) {
        const float y = __fadd_rn(__fdiv_rn((float)a, g), 0.5f);
        const uint32_t want = y >= 254.f ? 254u : (uint32_t)y;
        const uint32_t q = (a * (uint32_t)m + (1u << (kMulShift - 1))) >> kMulShift;
        ok = (q < 254u ? q : 254u) == want;
      }
      if (ok) found = m;
    }
  }
  mul[i] = found;
}

// The per-strip calibration word the clusterizers read, built once per upload:
//   bits 0-7   thr_ch:   channel limit, the largest ADC that is NOT active;
//   bits 8-15  thr_seed: seed limit, the largest ADC that is NOT a seed;
//   bits 16-23 gap:      the longest linking gap below the strip;
// stored beside noise^2 of the strip (binary32, rounded once; summed by the
// cluster threshold), so that the scan gathers both with one 8-byte load.
//
// Limits (section 2: a strip is active / a seed when its ADC is larger than the
// channel / seed threshold times its noise): with P = T x noise rounded once in
// binary32 (P >= 0), an integer ADC satisfies (float)adc > P exactly when adc >
// floor(P), since every ADC is exactly representable; so the limit is floor(P),
// capped at 255 (no 8-bit ADC exceeds it).  A bad strip is never active nor a
// seed: both limits are 255.
//
// Linking gap (a candidate continues over at most max_seq_holes consecutive
// inactive good strips and at most max_seq_bad consecutive bad strips): G(t) is
// the largest g such that, among strips t-g .. t-1 of the channel, every maximal
// run of bad strips is at most max_bad long and every maximal run of good strips
// at most max_holes long.  The strips between successive active strips a < t are
// all inactive, so they are linked exactly when their gap t-a-1 is at most G(t): a
// gap that is valid stays valid when shortened from below, and one longer than
// G(t) contains the strip t-G(t)-1 that breaks a limit.  One thread per strip walks
// down from t-1.  The byte stored is min(G(t) + 1, t) <= 255 (G(t) <= t), the limit
// the clusterizers compare tile keys against (see the comment below).
__global__ void k_calib_pack(const float* __restrict__ noise, const uint32_t* __restrict__ mask,
                             uint2* __restrict__ calq, uint64_t n_strips, float t_ch,
                             float t_seed, int max_holes, int max_bad) {
  const uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n_strips) return;
  const int t = (int)(s % kStrips);
  const uint32_t* m = mask + (s - (uint64_t)t) / 32;  // the channel's 8 mask words
  int g = 0, run = 0, prev = -1;
  for (int u = t - 1; u >= 0; --u) {
    const int b = (int)((m[u >> 5] >> (u & 31)) & 1u);
    run = b == prev ? run + 1 : 1;
    prev = b;
    if (run > (b ? max_bad : max_holes)) break;
    ++g;
  }
  const bool bad = (m[t >> 5] >> (t & 31)) & 1u;
  const float nz = noise[s];
  auto limit = [&](float thr) -> uint32_t {
    const float p = __fmul_rn(thr, nz);
    return p >= 255.f ? 255u : (uint32_t)p;  // truncation = floor for p >= 0
  };
  // linking limit of the tile key difference: strip t is linked to the previous
  // active strip a of its channel when t - a <= g + 1 (<= t always holds); an active
  // strip of an earlier channel is at least t + 1 keys below, so with
  // lim = min(g + 1, t) one unsigned compare, key - prev - 1 >= lim, marks a new
  // candidate in both cases
  const uint32_t gap = (uint32_t)(g + 1 < t ? g + 1 : t);
  const uint32_t word = bad ? (255u | (255u << 8) | (gap << 16)) : (limit(t_ch) | (limit(t_seed) << 8) | (gap << 16));
  calq[s] = make_uint2(word, __float_as_uint(__fmul_rn(nz, nz)));
}

// ---------------------------------------------------------------- launch helpers

// Raises a kernel's dynamic shared memory limit to what a launch needs and
// returns its CTAs per SM.  The limit only grows (per device and kernel), and the
// occupancy is looked up once per device, kernel, block size and shared memory
// size, so that repeated launches make no driver calls for either.
struct Prep {
  int dev;
  const void* fn;
  int block;
  size_t smem;
  int per_sm;
};
struct Limit {
  int dev;
  const void* fn;
  size_t smem;
};
std::mutex g_prep_mu;
std::vector<Prep> g_prep;
std::vector<Limit> g_limit;

cudaError_t prepare(const void* fn, int block, size_t smem, int* per_sm) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e) return e;
  std::lock_guard<std::mutex> lock(g_prep_mu);
  Limit* lim = nullptr;
  for (Limit& l : g_limit)
    if (l.dev == dev && l.fn == fn) lim = &l;
  if (!lim) {
    g_limit.push_back(Limit{dev, fn, 0});
    lim = &g_limit.back();
  }
  if (smem > lim->smem) {
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
    lim->smem = smem;
  }
  for (const Prep& p : g_prep)
    if (p.dev == dev && p.fn == fn && p.block == block && p.smem == smem) {
      *per_sm = p.per_sm;
      return cudaSuccess;
    }
  int n = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, block, smem))) return e;
  g_prep.push_back(Prep{dev, fn, block, smem, n});
  *per_sm = n;
  return cudaSuccess;
}

// The kernels' parameters with the stream's spill areas.
KParams with_spill(const KParams& kp, const Scratch& s) {
  KParams k = kp;
  k.spill = s.spill;
  k.spill_warps = (uint32_t)s.spill_warps;
  return k;
}

// Launches `k` with programmatic stream serialization: it may start while the
// kernel before it on the stream drains, and waits for it with pdl_wait().
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*k)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                       Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, std::forward<Args>(args)...);
}

// k_stream's amplitude arguments: none unless the caller asked for them.
cs::Amps amp_args(const sst_clusters& out, const Scratch& s) {
  cs::Amps a;
  if (!out.amp) return a;
  a.spill = s.amp_spill;
  a.bytes = s.amp_stage;
  a.first = s.stage_amp;
  a.off = out.amp_off;
  a.cap = out.amp_capacity;
  a.alloc = s.amp_alloc;
  a.seg_cnt = s.seg_amp_cnt;
  a.seg_start = s.seg_amp_start;
  return a;
}

// The shared state of a launch of one CTA per FED of n_events events, under the next tag
// of l (the last for a launch that a graph may replay).  The state is cleared before a
// captured launch and when half of the tags have gone round: a word keeps its tag at most
// that long, and work that wrongly overlapped a clearing is cleared away by the next one
// before its tag is due again.
cudaError_t shared_state(const Scratch& s, LookState& l, uint32_t n_events, uint32_t n_feds, cudaStream_t st,
                         ev::Shared* sh) {
  const size_t items = (size_t)n_events * n_feds;
  if (!l.words || n_events > l.events || items > l.items) return cudaErrorInvalidValue;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(st, &cs);
  if (e) return e;
  constexpr uint32_t kTurn = LookState::kTags - 2;
  uint32_t tag = LookState::kTags - 1;
  bool clear = true;
  if (cs == cudaStreamCaptureStatusNone) {
    const uint32_t n = __atomic_fetch_add(&l.launches, 1u, __ATOMIC_RELAXED) % kTurn;  // (0 when the count wraps, too)
    tag = n + 1;
    clear = n % (kTurn / 2) == 0;
  }
  if (clear && (e = cudaMemsetAsync(l.words, 0, LookState::words_for(l.events, l.items) * sizeof(*l.words), st))) return e;
  sh->ticket = reinterpret_cast<uint32_t*>(l.words) + tag;
  sh->lb = l.words + LookState::kTags / 2;
  sh->pre = sh->lb + l.items;
  sh->late = reinterpret_cast<uint32_t*>(sh->pre + 4 * (l.items / 1024 + 1));
  sh->st = sh->late + (l.events + 1) / 2 * 2;
  sh->n_items = (uint32_t)items;
  sh->n_feds = n_feds;
  sh->tag = tag;
  sh->spin_limit = s.lb_spin_limit ? s.lb_spin_limit : kLbSpinLimit;
  sh->withhold = s.lb_withhold;
  return cudaSuccess;
}

// Launches kernel k of n_events x n_feds CTAs with the shared state as its last or, in
// k_unpack, last but one argument (bind makes the call).
template <typename Bind>
cudaError_t launch_feds(const void* fn, size_t smem, const Scratch& s, LookState& l, uint32_t n_events,
                        uint32_t n_feds, cudaStream_t st, Bind bind) {
  int per_sm = 0;
  ev::Shared sh;
  cudaError_t e = prepare(fn, ev::kThreads, smem, &per_sm);
  if (!e) e = shared_state(s, l, n_events, n_feds, st, &sh);
  return e ? e : bind(sh);
}

template <int TILE>
cudaError_t launch_unpack_t(const uint8_t* raw, uint64_t raw_bytes, const uint32_t* fed_len, uint32_t n_feds,
                            const sst_digis& out, Scratch& s, const Shape& shape, cudaStream_t st) {
  const size_t sm = sizeof(ev::Shm<TILE, false>);
  return launch_feds((const void*)k_unpack<TILE>, sm, s, s.look_unpack, 1, n_feds, st, [&](ev::Shared& sh) {
    return launch_pdl(k_unpack<TILE>, n_feds, (unsigned)ev::kThreads, sm, st, raw, raw_bytes, fed_len, out, sh,
                      shape.lanes);
  });
}

template <int TILE>
cudaError_t launch_event_t(const uint8_t* raw, const uint64_t* event_off, const uint64_t* event_end,
                           const uint32_t* fed_len, uint32_t n_events, uint32_t n_feds, const uint64_t* clu_off,
                           const sst_clusters& out, sst_event_status* status, const KParams& kp, Scratch& s,
                           cudaStream_t st, uint64_t* pack_off) {
  const size_t sm = sizeof(ev::Shm<TILE, true>);
  auto* k = out.amp ? k_event<true, TILE> : k_event<false, TILE>;
  return launch_feds((const void*)k, sm, s, s.look_event, n_events, n_feds, st, [&](ev::Shared& sh) {
    return launch_pdl(k, n_events * n_feds, (unsigned)ev::kThreads, sm, st, raw, event_off, event_end, fed_len,
                      n_events, clu_off, out, status, with_spill(kp, s), pack_off, sh);
  });
}

// Whether `feds` CTAs of k_cluster (or k_event) fit the GPU at once with the larger tile.  A
// FED of more than a tile of digis goes through the steps chunk by chunk.  k_cluster, 440 FEDs,
// unpacking included: 31.4 -> 28.8 us (fewer registers spilled), densities a hundredfold apart
// 73.7 -> 69.2, 4,700 digis a FED 106 -> 99; but 500 FEDs, two waves then, 32 -> 39.  k_event,
// one event of 440 FEDs 26.1 -> 25.1, a hundredfold apart 99 -> 83, 2,750 digis a FED 60 -> 37.
cudaError_t large_tile(const void* fn, size_t feds, int n_sm, bool* large) {
  int per_sm = 0;
  const cudaError_t e = prepare(fn, ev::kThreads, sizeof(ev::Shm<kEvTileLarge, true>), &per_sm);
  *large = !e && feds <= (size_t)n_sm * per_sm;
  return e;
}

// Which kernel a batch takes, by its events, FEDs and FED records (events x FEDs).  Times
// in us a batch; "skewed": the FEDs' densities differ up to a hundredfold either way.
//   k_event (a CTA per record, one launch) has the shortest critical path but the least
//   throughput, and a long FED holds it up most: 440 FEDs x 1 event 25 (k_stream_fed 31),
//   x 2 50 (41); with amplitudes x 2 57 (54), x 3 skewed 436 (k_stream_fed from here on).
//   k_stream pays for its tiles: while they all fit the GPU at once (up to 76 FEDs) it is
//   the fastest from 100 records on (13 FEDs x 17 events 18.6 against k_event's 22.5,
//   skewed 37 against 112; 61 x 2 17.7 and 20.6), but a single FED has 8 tiles (1 x 120:
//   24 and 18); beyond, from 1,500 records of 10 events and more on (200 x 10 54,
//   k_stream_fed 59; 120 x 13 43 and 45; 100 x 12 40 and 36; 440 x 9 99 and 97; 440 x 8 105
//   and 87), or of 16 events; where the calibration is larger than the L2 (above 640 FEDs)
//   every tile comes from DRAM: from 24 events on (1000 x 24 276 and 290; 1000 x 16 242 and
//   221; 1000 x 4 168 and 111; 4096 x 1 474 and 148).
// The densities are not known here, and no line is best for all: against one warp per pair of
// FE units (the kernel before these) the choice loses 100 x 6 skewed 95 -> 98 and 77 x 12
// skewed 113 -> 121 (tiles: 53 and 52, but 37 and 36 for 27 and 32 when they are alike),
// 200 x 6 skewed 105 -> 117 (four units a warp; two: 81, but 43 for 39 when alike), 200 x 9 47
// -> 52 (two units a warp; four: 45, but 116 for 88 when skewed), 440 x 8 with amplitudes 114
// -> 123 (204 -> 170 when dense, 250 -> 216 when skewed).
// A batch read in place from pinned host memory is bound by the link, which a warp's
// contiguous piece of four FE units (1.4 KB) loads better than the tiles' single units:
// 440 FEDs x 16 | 32 | 64 | 128 events 153 | 253 | 448 | 853 us with k_stream_fed, 150 | 267
// | 500 | 965 with k_stream (two units: 147 | 249 | 450 | 866); served, 87 | 93 | 101 | 104 k
// events/s against 79 | 80 | 84 | 87 k (two units: 87 | 90 | 98 | 99 k).  Fetching ahead to
// L2 does not pay there (k_stream without it: 83 | 84 | 88 | 90 k).
constexpr uint32_t kEventRecords = 100, kEventRecordsOneFed = 240, kEventRecordsWide = 700, kEventRecordsAmps = 850;
static_assert(kEventRecords <= kEventRecordsMost && kEventRecordsOneFed <= kEventRecordsMost &&
                  kEventRecordsWide <= kEventRecordsMost && kEventRecordsAmps <= kEventRecordsMost &&
                  kEventRecordsMost <= ev::kLbBlock,
              "k_event's shared state has room for the records it takes, in one look-back block");
constexpr uint32_t kTileEvents = 10, kTileEventsFew = 16, kTileRecordsFew = 1500;
constexpr uint32_t kTileEventsMany = 24, kTileFedsMany = 640;
constexpr uint32_t kTileChunk = 32, kTileChunkMin = 8;

// How a batch is launched.
struct Plan {
  enum Kind { kFeds, kUnits, kTiles } kind = kFeds;  // k_event, k_stream_fed, k_stream
  int grid = 0, block = 0, resident = 0;
  size_t smem = 0;
  uint32_t segs_per_fed = kFe;     // segments of the staging buffer per FED and event
  bool large = false;              // kFeds: the larger tile
  uint32_t units = 0;              // kUnits: FE units per warp
  bool link = false;               // kUnits: the records are read in place from host memory
  uint32_t chunk = 0, per_warp = 0;  // kTiles: events per item, and per warp of it
};

template <int W, int U>
cudaError_t plan_tiles(const Shape& sh, uint32_t n_events, uint32_t n_feds, int n_sm, Plan* p) {
  p->block = W * 32;
  p->smem = sizeof(uint2) * (3 * W / 2) * kStrips + W * sizeof(cs::WarpT<U>);
  p->segs_per_fed = kFe * (8 / W);
  int per_sm = 0;
  cudaError_t e = prepare((const void*)k_stream<false, W, U>, p->block, p->smem, &per_sm);
  if (e) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const size_t per = sh.ctas_per_sm < kMaxWarpsPerSm / W ? sh.ctas_per_sm : kMaxWarpsPerSm / W;
  const size_t ctas = (size_t)n_sm * per, fit = (size_t)n_sm * per_sm, tiles = (size_t)n_feds * p->segs_per_fed;
  // Few tiles: their events are shared out, down to kTileChunk at a time for a second
  // wave and to kTileChunkMin while that is one wave at most (2 FEDs x 147 events: 45 us
  // with chunks of 37, 33 of 19, 27 of 10; but 3 FEDs x 256: 35 with 384 items, 46 with 768).
  uint32_t chunks = 1;
  auto halves = [&] { return (n_events + 2 * chunks - 1) / (2 * chunks); };  // events of a chunk with twice as many
  while ((tiles * chunks < 2 * fit && halves() >= kTileChunk) || (2 * tiles * chunks <= fit && halves() >= kTileChunkMin))
    chunks *= 2;
  p->chunk = (n_events + chunks - 1) / chunks;
  const uint32_t passes = (p->chunk + W * 32 - 1) / (W * 32);  // at most 32 events, a lane each, per warp and pass
  p->per_warp = (p->chunk + W * passes - 1) / (W * passes);
  const size_t items = tiles * ((n_events + p->chunk - 1) / p->chunk);
  p->grid = (int)(ctas < items ? ctas : items);
  p->resident = (int)(fit < (size_t)p->grid ? fit : (size_t)p->grid);
  return cudaSuccess;
}

cudaError_t plan_batch(const Shape& sh, uint32_t n_events, uint32_t n_feds, bool amps, bool in_place, int n_sm,
                       Plan* p) {
  const size_t records = (size_t)n_events * n_feds;
  const bool one_wave = (size_t)n_feds * kFe <= (size_t)n_sm * 4;  // the tiles fit the GPU at once
  const bool tiles = one_wave || n_events >= (n_feds > kTileFedsMany        ? kTileEventsMany
                                              : records < kTileRecordsFew ? kTileEventsFew
                                                                          : kTileEvents);
  if (records < (one_wave ? n_feds > 1 ? kEventRecords : kEventRecordsOneFed
                 : amps ? kEventRecordsAmps : kEventRecordsWide) &&
      (one_wave || !tiles)) {
    p->kind = Plan::kFeds;
    p->grid = (int)records;
    p->block = ev::kThreads;
    const cudaError_t e = large_tile((const void*)k_event<false, kEvTileLarge>, records, n_sm, &p->large);
    p->smem = p->large ? sizeof(ev::Shm<kEvTileLarge, true>) : sizeof(ev::Shm<kEvTile, true>);
    return e;
  }
  if (tiles && !in_place) {
    p->kind = Plan::kTiles;
    auto* f = sh.block == 128 ? (sh.units == 1 ? plan_tiles<4, 1> : plan_tiles<4, 2>)
                              : (sh.units == 1 ? plan_tiles<8, 1> : plan_tiles<8, 2>);
    return f(sh, n_events, n_feds, n_sm, p);
  }
  p->kind = Plan::kUnits;
  p->link = in_place;
  p->block = kFedWarps * 32;
  p->smem = kFedWarps * sizeof(FedWarp);
  int per_sm = 0;
  cudaError_t e = prepare((const void*)k_stream_fed<false, false>, p->block, p->smem, &per_sm);
  if (e) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const size_t per = sh.ctas_per_sm < per_sm ? sh.ctas_per_sm : per_sm, ctas = (size_t)n_sm * per;
  // FE units per warp: as few as give every warp one item, half a FED's at most (48
  // channels); two (24 channels, evener shares) where halves fill more than two thirds of
  // a wave: 440 FEDs x 3 events 56.6 with halves, 57.3 with quarters, but 256 and 161
  // when the FEDs' densities differ a hundredfold; 440 x 5 77 and 69; 150 x 8 36 and 42.
  // Halves again from 8,500 records on: 1000 x 8 153 and 174 with quarters, but 236 and 197
  // skewed; 1000 x 10 175 and 207, 255 and 227; 2000 x 16 401 and 542, 491 and 542.
  p->units = 1;
  while (p->units < kFe / 2 && records * (kFe / p->units) > ctas * kFedWarps) p->units *= 2;
  if (records * 3 > ctas * kFedWarps) p->units = in_place || records > 8500 ? 4 : 2;
  const size_t need = (records * (kFe / p->units) + kFedWarps - 1) / kFedWarps;
  p->grid = (int)(ctas < need ? ctas : need);
  p->resident = p->grid;
  return cudaSuccess;
}

template <bool AMP, int W, int U>
cudaError_t launch_tiles(const Plan& p, const uint8_t* raw, uint32_t n_events, uint32_t n_feds,
                         const uint64_t* clu_off, uint64_t out_cap, sst_event_status* status, const KParams& kp,
                         const Scratch& s, const cs::Amps& am, cudaStream_t st) {
  int per_sm = 0;
  cudaError_t e = prepare((const void*)k_stream<AMP, W, U>, p.block, p.smem, &per_sm);
  if (e) return e;
  return launch_pdl(k_stream<AMP, W, U>, (unsigned)p.grid, (unsigned)p.block, p.smem, st, raw,
                    (const uint64_t*)s.fed_off, n_events, n_feds, clu_off, out_cap, status, kp, s.stage, s.ev_alloc,
                    s.fed_cnt, s.fed_start, s.tickets, (const uint2*)s.unit_desc, p.chunk, p.per_warp,
                    (uint32_t)p.resident, am);
}

template <bool AMP>
cudaError_t launch_stream(const Plan& p, const Shape& sh, const uint8_t* raw, uint32_t n_events, uint32_t n_feds,
                          const uint64_t* clu_off, uint64_t out_cap, sst_event_status* status, const KParams& kp,
                          const Scratch& s, const cs::Amps& am, cudaStream_t st) {
  if ((size_t)p.grid * (p.block / 32) > s.spill_warps) return cudaErrorInvalidConfiguration;
  const KParams kps = with_spill(kp, s);
  if (p.kind == Plan::kTiles) {
    auto* f = sh.block == 128 ? (sh.units == 1 ? launch_tiles<AMP, 4, 1> : launch_tiles<AMP, 4, 2>)
                              : (sh.units == 1 ? launch_tiles<AMP, 8, 1> : launch_tiles<AMP, 8, 2>);
    return f(p, raw, n_events, n_feds, clu_off, out_cap, status, kps, s, am, st);
  }
  int per_sm = 0;
  auto* k = !AMP && p.link ? k_stream_fed<false, true> : k_stream_fed<AMP, false>;
  cudaError_t e = prepare((const void*)k, p.block, p.smem, &per_sm);
  if (e) return e;
  return launch_pdl(k, (unsigned)p.grid, (unsigned)p.block, p.smem, st, raw,
                    (const uint64_t*)s.fed_off, n_events, n_feds, clu_off, out_cap, status, kps, s.stage, s.ev_alloc,
                    s.fed_cnt, s.fed_start, s.tickets, (const uint2*)s.unit_desc, p.units, am);
}

// k_stream's per-event cluster order and the copy into the caller's SoA.  chans:
// channels per segment.
cudaError_t launch_order(const uint64_t* clu_off, uint32_t n_events, uint32_t n_segs, const sst_clusters& out,
                         sst_event_status* status, const Scratch& s, uint64_t* pack_off, uint32_t chans,
                         const cs::Amps& am, cudaStream_t st) {
  cudaError_t e;
  if (pack_off) {
    k_clu_scan<<<n_events, 1024, 0, st>>>(s.fed_cnt, n_segs, status, pack_off, s.tickets + 1);
    if ((e = cudaGetLastError())) return e;
  }
  // 128 segments per CTA; 32 or 16 when that would give a small grid, so that enough
  // CTAs share the copy
  const uint64_t all = (uint64_t)n_events * n_segs;
  const uint32_t per = all >= 128 * 1000 ? 128u : all >= 32 * 500 ? 32u : 16u;
  const uint32_t cpe = (n_segs + per - 1) / per;
  auto* k = am.bytes ? (per == 128 ? k_order<128, true> : per == 32 ? k_order<32, true> : k_order<16, true>)
                     : (per == 128 ? k_order<128, false> : per == 32 ? k_order<32, false> : k_order<16, false>);
  return launch_pdl(k, (unsigned)((uint64_t)n_events * cpe), 256u, 0, st,
                    (const uint2*)s.stage, clu_off, (const uint64_t*)pack_off, (const uint32_t*)s.fed_cnt,
                    (const uint32_t*)s.fed_start, n_segs, cpe, out, status, chans, am);
}

}  // namespace

// ---------------------------------------------------------------- host side

Shape default_shape() { return Shape{256, 2048, 2, 4, 0, 2}; }

bool shape_valid(const Shape& s) {
  const bool blk = s.block == 128 || s.block == 256;
  const bool til = s.tile == 1024 || s.tile == 2048 || s.tile == 4096;
  const bool ln = s.lanes == 1 || s.lanes == 2 || s.lanes == 4 || s.lanes == 8 || s.lanes == 16 || s.lanes == 32;
  return blk && til && ln && s.ctas_per_sm >= 1 && s.ctas_per_sm <= 8 && s.host_chunk >= 0 && s.host_chunk <= 4096 &&
         (s.units == 1 || s.units == 2);
}

cudaError_t batch_launch_info(const Shape& sh, uint32_t n_events, uint32_t n_feds, int n_sm, int* grid, size_t* smem,
                              int* block, int* items_per_fed) {
  Plan p;
  const bool amps = false;
  const cudaError_t e = plan_batch(sh, n_events, n_feds, amps, false, n_sm, &p);
  if (e) return e;
  *grid = p.grid;
  *block = p.block;
  *smem = p.smem;
  *items_per_fed = p.kind == Plan::kTiles ? kFe / sh.units : p.kind == Plan::kUnits ? (int)(kFe / p.units) : 1;
  return cudaSuccess;
}

cudaError_t launch_unpack(const uint8_t* raw, uint64_t raw_bytes, const uint32_t* fed_len, uint32_t n_feds,
                          const sst_digis& out, Scratch& s, const Shape& sh, cudaStream_t st) {
  switch (sh.tile) {
    case 1024: return launch_unpack_t<1024>(raw, raw_bytes, fed_len, n_feds, out, s, sh, st);
    case 2048: return launch_unpack_t<2048>(raw, raw_bytes, fed_len, n_feds, out, s, sh, st);
    case 4096: return launch_unpack_t<4096>(raw, raw_bytes, fed_len, n_feds, out, s, sh, st);
    default: return cudaErrorInvalidValue;
  }
}

template <int TILE>
static cudaError_t launch_cluster_t(const sst_digis& in, uint32_t n_feds, const sst_clusters& out, const KParams& kp,
                                    Scratch& s, cudaStream_t st) {
  const size_t sm = sizeof(ev::Shm<TILE, true>);
  auto* k = out.amp ? k_cluster<true, TILE> : k_cluster<false, TILE>;
  return launch_feds((const void*)k, sm, s, s.look_cluster, 1, n_feds, st, [&](ev::Shared& sh) {
    return launch_pdl(k, n_feds, (unsigned)ev::kThreads, sm, st, in, with_spill(kp, s), out, sh);
  });
}

cudaError_t launch_cluster(const sst_digis& in, uint32_t n_feds, const sst_clusters& out, const KParams& kp,
                           Scratch& s, int n_sm, cudaStream_t st) {
  bool large = false;
  const cudaError_t e = large_tile((const void*)k_cluster<false, kEvTileLarge>, n_feds, n_sm, &large);
  if (e) return e;
  return large ? launch_cluster_t<kEvTileLarge>(in, n_feds, out, kp, s, st)
               : launch_cluster_t<kEvTile>(in, n_feds, out, kp, s, st);
}

cudaError_t launch_batch(const uint8_t* raw, const uint64_t* event_off, const uint32_t* fed_len, uint32_t n_events,
                         uint32_t n_feds, const uint64_t* clu_off, const sst_clusters& out, sst_event_status* status,
                         const KParams& kp, Scratch& s, const Shape& sh, int n_sm, cudaStream_t st,
                         uint64_t* pack_off, cudaEvent_t ev_begin, cudaEvent_t ev_end, const uint64_t* event_end) {
  Plan p;
  const bool amps = out.amp != nullptr;
  cudaError_t e = plan_batch(sh, n_events, n_feds, amps, event_end != nullptr, n_sm, &p);
  if (e) return e;
  if (p.kind == Plan::kFeds) {
    if (ev_begin && (e = cudaEventRecord(ev_begin, st))) return e;
    e = (p.large ? launch_event_t<kEvTileLarge> : launch_event_t<kEvTile>)(raw, event_off, event_end, fed_len, n_events,
                                                                           n_feds, clu_off, out, status, kp, s, st,
                                                                           pack_off);
    if (e) return e;
    return ev_end ? cudaEventRecord(ev_end, st) : cudaSuccess;
  }
  const uint32_t cpe = (n_feds + kFedScanThreads - 1) / kFedScanThreads;
  k_fed_scan<<<(unsigned)((uint64_t)n_events * cpe), kFedScanThreads, 0, st>>>(
      event_off, event_end, fed_len, n_feds, cpe, s.fed_off, status, s.ev_alloc, s.tickets, raw, s.unit_desc,
      out.amp ? s.amp_alloc : nullptr);
  if ((e = cudaGetLastError())) return e;
  if (ev_begin && (e = cudaEventRecord(ev_begin, st))) return e;
  const cs::Amps am = amp_args(out, s);
  e = (out.amp ? launch_stream<true> : launch_stream<false>)(p, sh, raw, n_events, n_feds, clu_off, out.capacity,
                                                             status, kp, s, am, st);
  if (e) return e;
  if (ev_end && (e = cudaEventRecord(ev_end, st))) return e;
  return launch_order(clu_off, n_events, n_feds * p.segs_per_fed, out, status, s, pack_off,
                      (uint32_t)kCh / p.segs_per_fed, am, st);
}

cudaError_t rebase_amp_first(uint32_t* amp_first, const uint64_t* count, uint32_t base, int n_sm, cudaStream_t st) {
  k_rebase_amp<<<(unsigned)(n_sm > 0 ? n_sm * 2 : 128), 256, 0, st>>>(amp_first, count, base);
  return cudaGetLastError();
}

cudaError_t build_badmask(const uint8_t* bad_dev, uint32_t* mask_dev, uint64_t n_strips, cudaStream_t st) {
  const uint64_t words = n_strips / 32;
  k_badmask<<<(unsigned)((words + 255) / 256), 256, 0, st>>>(bad_dev, mask_dev, words);
  return cudaGetLastError();
}

cudaError_t build_gain(const float* gain_dev, int32_t* mul_dev, uint32_t n_apv, cudaStream_t st) {
  k_gain_pack<<<(n_apv + 127) / 128, 128, 0, st>>>(gain_dev, mul_dev, n_apv);
  return cudaGetLastError();
}

cudaError_t build_calib(const float* noise_dev, const uint32_t* mask_dev, uint2* calq_dev, uint64_t n_strips,
                        const sst_params& p, cudaStream_t st) {
  k_calib_pack<<<(unsigned)((n_strips + 255) / 256), 256, 0, st>>>(noise_dev, mask_dev, calq_dev, n_strips,
                                                                   p.t_channel, p.t_seed, p.max_seq_holes,
                                                                   p.max_seq_bad);
  return cudaGetLastError();
}

}  // namespace sst

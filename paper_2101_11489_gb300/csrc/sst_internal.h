// sst_internal.h -- internal declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "../../include/sst.h"

namespace sst {

constexpr int kCh = SST_CH_PER_FED;          // channels per FED
constexpr int kStrips = SST_STRIPS_PER_CH;   // strips per channel (module)
constexpr int kFe = SST_FE_PER_FED;          // FE units per FED
constexpr int kChPerFe = SST_CH_PER_FE;      // channels per FE unit
constexpr int kApv = SST_STRIPS_PER_APV;     // strips per APV
constexpr int kHdr = SST_FED_HEADER_BYTES;   // FED header bytes
constexpr int kFedStrips = kCh * kStrips;    // 24,576 strips per FED
constexpr int kMulShift = 22;                // fixed-point charge multipliers: binary places
constexpr int kMaskWords = kStrips / 32;     // 8 words of 32 strips per channel

// Calibration and thresholds as the kernels see them.  The per-strip tables are
// built on the device at calibration upload (k_calib_pack) from the noise, the
// bad-strip flags and the parameters, the per-APV multipliers from the gains
// (k_gain_pack).
struct KParams {
  float t_cluster;
  int max_adj;
  const uint2* calq;        // [n_strips]: {thr_ch | thr_seed << 8 | gap << 16, noise^2 (binary32 bits)}
                            // (see k_calib_pack); one 8-byte load per recorded strip
  const uint32_t* badmask;  // [n_strips / 32], bit (s & 31) of word s / 32
  const int32_t* mul;       // [n_strips / 128]: per APV, the fixed-point charge multiplier, or the bits of -gain (k_gain_pack)
  uint4* spill = nullptr;   // k_stream: candidate lists (one per warp of the grid, kSpillRecords records each)
  uint32_t spill_warps = 0; // warps that have one
};

// Launch shape of the kernels.
struct Shape {
  int block;        // batched kernel: threads per CTA
  int tile;         // per-event unpack kernel: digis per on-chip tile
  int lanes;        // per-event unpack kernel: lanes per channel when copying runs
  int ctas_per_sm;  // batched kernel: persistent CTAs per SM
  int host_chunk = 0;  // events per chunk of sst_batch_host (0: automatic)
  int units = 2;       // batched kernel: FE units per warp work item (1 or 2)
};

// What the CTAs of a one-CTA-per-FED launch share (ev::Shared).  Every word that a launch
// reads carries the launch's tag, and every tag has a ticket counter of its own, so that
// no launch depends on what the one before it left or cleared: 0 marks cleared words,
// ordinary launches take 1 .. kTags - 2 in turn, launches captured into a graph (whose
// replays are not seen on the host) the last, and clear the state themselves, ahead.
// Each kind of launch has a state of its own: an unpacking and a clustering call of one
// context may overlap on two streams.  Allocated once, so that captured launches keep it.
struct LookState {
  static constexpr uint32_t kTags = 1024;
  unsigned long long* words = nullptr;
  size_t events = 0, items = 0;  // most events, and FED records over all of them
  uint32_t launches = 1;         // counts ordinary launches (atomically); the first finds cleared words
  // tickets, a count per FED record, four sums per 1024 of them, a word of 32 bits per event and per record
  static constexpr size_t words_for(size_t events, size_t items) {
    return kTags / 2 + items + 4 * (items / 1024 + 1) + (events + 1) / 2 + (items + 1) / 2;
  }
};
constexpr uint32_t kEventRecordsMost = 850;  // FED records of a batch that k_event takes: fewer than this

// Device scratch for one stream of work, owned by a context (or by one server
// stream): the state shared by the CTAs of the one-CTA-per-FED kernels, work tickets,
// and the many-event kernel's FED offsets, cluster bookkeeping and staging buffer.
struct Scratch {
  LookState look_unpack, look_cluster;  // the per-event calls' (contexts only)
  LookState look_event;                 // k_event's
  uint64_t* fed_off = nullptr;       // absolute byte offset per (event, FED)
  uint32_t* fed_cnt = nullptr;       // clusters found per segment (event, FE unit or half of one)
  uint32_t* fed_start = nullptr;     // staging offset per segment, within its event's slice
  uint2* unit_desc = nullptr;        // per (event, FED, FE unit): offset in the FED record, length | status
  size_t items_cap = 0;
  uint32_t* ev_alloc = nullptr;      // staging allocation counter per event (counter_at)
  size_t ev_cap = 0;
  uint2* stage = nullptr;            // staged cluster records (8 bytes each)
  size_t stage_cap = 0;
  uint32_t* tickets = nullptr;       // [16]: [0] k_stream's tiles, [1] k_clu_scan's CTAs done
  uint4* spill = nullptr;            // per warp of k_stream, kSpillRecords candidate records
  size_t spill_warps = 0;            // warps that have them
  // clusters with amplitudes (k_stream)
  uint8_t* amp_stage = nullptr;      // staged amplitudes, sliced per event like the output
  size_t amp_stage_cap = 0;
  uint32_t* stage_amp = nullptr;     // per staged cluster: its first amplitude within its segment
  size_t stage_amp_cap = 0;
  uint32_t* amp_alloc = nullptr;     // amplitude allocation counter per event (counter_at)
  size_t amp_ev_cap = 0;
  uint32_t* seg_amp_cnt = nullptr;   // amplitudes per segment; 0 when they did not fit
  uint32_t* seg_amp_start = nullptr; // their offset in the event's slice, or kNoAmp
  size_t amp_items_cap = 0;
  uint32_t* amp_spill = nullptr;     // per warp that has a spill area, kAmpSpill words
  size_t amp_spill_warps = 0;
  uint32_t lb_spin_limit = 0;        // polls before a look-back wait gives up (0: the default, about a second)
  int32_t lb_withhold = -1;          // failure tests: the FED (of a batch's first event) that never publishes its counts (-1: none)
};
// Where event e's allocation counter is: up to 1,024 events have a 128-byte line each, so
// that the warps' additions do not queue at one line of L2, or at two that share a slice.
// (12 events of 100 FEDs with amplitudes: 51 us; with adjacent counters 52 to 58 us, by
// the addresses that the arrays happened to have.)
__host__ __device__ constexpr size_t counter_at(uint32_t e) {
  return ((size_t)(e >> 15) << 15) + (e & 1023u) * 32u + ((e >> 10) & 31u);
}
constexpr size_t counters_for(size_t events) { return (events + 32767) / 32768 * 32768; }
constexpr uint32_t kNoAmp = 0xFFFFFFFFu;
constexpr uint32_t kSpillRecords = 1608;  // records per warp spill area (25 KiB)
constexpr uint32_t kAmpSpill = kSpillRecords + 128;  // words per warp beside them for clusters with amplitudes
constexpr int kMaxWarpsPerSm = 32;        // resident warps of the batched kernel per SM (its register use)

// Grid, block, shared memory per CTA and work items per FED of the batched kernel's
// launch for a shape and batch (the occupancy look-up may call the driver once).
cudaError_t batch_launch_info(const Shape& sh, uint32_t n_events, uint32_t n_feds, int n_sm, int* grid, size_t* smem,
                              int* block, int* items_per_fed);
// Chunks sst_batch_host cuts a batch of n_events into (tuned: events per chunk, 0 = automatic).
uint32_t host_chunks(uint32_t n_events, int tuned);
Shape default_shape();
bool shape_valid(const Shape& s);

// Kernel launchers (sst_kernels.cu).  They only enqueue work on `st`.
cudaError_t launch_unpack(const uint8_t* raw, uint64_t raw_bytes, const uint32_t* fed_len, uint32_t n_feds,
                          const sst_digis& out, Scratch& s, const Shape& sh, cudaStream_t st);
cudaError_t launch_cluster(const sst_digis& in, uint32_t n_feds, const sst_clusters& out, const KParams& kp,
                           Scratch& s, int n_sm, cudaStream_t st);
// Kernels launched per batched call: k_event alone for the fewest events; else k_fed_scan,
// k_stream or k_stream_fed, and k_order (before it k_clu_scan for packed output).
// Batched unpack + cluster.  Event e's clusters are written to the slice [clu_off[e], clu_off[e+1]) of `out` (bounded by
// out.capacity).  With pack_off (device, n_events + 1 values) the events' clusters
// are written back to back instead, event e from pack_off[e], which the launch
// computes.  With event_end (device, n_events values) event e's bytes are
// [event_off[e], event_end[e]) of raw, so that the events need not follow one
// another (raw may then be pinned host memory read in place).
cudaError_t launch_batch(const uint8_t* raw, const uint64_t* event_off, const uint32_t* fed_len, uint32_t n_events,
                         uint32_t n_feds, const uint64_t* clu_off, const sst_clusters& out, sst_event_status* status,
                         const KParams& kp, Scratch& s, const Shape& sh, int n_sm, cudaStream_t st,
                         uint64_t* pack_off = nullptr, cudaEvent_t ev_begin = nullptr, cudaEvent_t ev_end = nullptr,
                         const uint64_t* event_end = nullptr);
cudaError_t build_badmask(const uint8_t* bad_dev, uint32_t* mask_dev, uint64_t n_strips, cudaStream_t st);
// Adds base to the first *count (device) values of amp_first, kNoAmp excepted.
cudaError_t rebase_amp_first(uint32_t* amp_first, const uint64_t* count, uint32_t base, int n_sm, cudaStream_t st);
cudaError_t build_gain(const float* gain_dev, int32_t* mul_dev, uint32_t n_apv, cudaStream_t st);
cudaError_t build_calib(const float* noise_dev, const uint32_t* mask_dev, uint2* calq_dev,
                        uint64_t n_strips, const sst_params& p, cudaStream_t st);

}  // namespace sst

struct sst_server;
struct sst_host_pipe;

struct sst_ctx {
  int device = 0;
  uint32_t n_feds = 0;
  int n_sm = 0;
  bool has_calib = false;
  sst_params params{};
  uint2* calq = nullptr;       // per strip: channel and seed thresholds as ADC limits and linking gap; noise^2
  uint32_t* badmask = nullptr;
  int32_t* mul = nullptr;      // per APV: fixed-point charge multiplier or the bits of -gain
  sst::Scratch scratch;
  sst::Shape shape{};
  std::string err;
  std::mutex mu;
  sst_server* server = nullptr;
  sst_host_pipe* pipe = nullptr;  // streams and arenas of sst_batch_host, made on first use
  float* pitch = nullptr;         // strip pitch per module (sst_pitch_upload), or null
  bool profiling = false;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> prof_events;  // recorded launches
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> prof_free;    // reusable pairs
};

namespace sst {
sst_status set_err(sst_ctx* c, sst_status code, const std::string& msg);
sst_status cuda_err(sst_ctx* c, cudaError_t e, const char* where);
KParams kparams(const sst_ctx* c);
cudaError_t ensure_scratch(Scratch& s, size_t items, size_t events, size_t stage_records);
// Memory for launches of up to `events` events of `items` FED records in all, once.
cudaError_t ensure_look(LookState& l, size_t events, size_t items);
// Candidate lists for `warps` warps of k_stream; grows only.
cudaError_t ensure_spill(Scratch& s, size_t warps);
// What k_stream needs for amplitudes beside the above, for a launch of that size (after
// ensure_spill); grows only, and only when that launch needs it.
cudaError_t ensure_amp_scratch(Scratch& s, size_t items, size_t events, size_t stage_records, size_t amp_bytes);
bool amp_scratch_fits(const Scratch& s, size_t items, size_t events, size_t stage_records, size_t amp_bytes);
void free_scratch(Scratch& s);
void free_host_pipe(sst_ctx* ctx);

// Makes `dev` current for the guard's lifetime.
struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    if (prev != dev) cudaSetDevice(dev);
  }
  ~DeviceGuard() {
    int cur = -1;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
  }
};
}  // namespace sst

// sst_event.cuh -- one CTA per FED, output in order by the CTA itself: the per-event
// kernels (unpack to a digi SoA, cluster a digi SoA) and the kernel of the smallest
// batches (both steps in one pass, the digis never leaving the chip).
//
// A single event has 440 FEDs: what bounds these kernels is the chain of dependent
// steps of one FED, so every step is spread over the CTA's threads and everything
// around the step is kept short: no prologue (a CTA sums the FED lengths before its
// own), no ordering pass (a CTA sums the counts that the FEDs before it publish) and
// no clearing between launches (what a launch reads carries its tag).  An event
// of 440 FEDs took 48 us in four launches and a memset, a warp per FE unit; it takes 30
// in two (8 FEDs: 29 and 17; the allocation-free unpack of 440 FEDs: 21 and 11).
//
// Included by sst_kernels.cu only, inside its namespace.
#pragma once

namespace ev {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kFedBuf = 8192;      // bytes of FED record that have run slots (larger ones are staged without, if at all)
constexpr int kRunSlots = (kFedBuf + 2) / 3;  // a run header takes at least 3 bytes with its ADC
constexpr uint32_t kFedClusters = kCh * kStrips / 2;  // most clusters of a FED whose strips ascend
constexpr uint32_t kLbBlock = 1024;  // FEDs whose counts a CTA sums one by one
constexpr uint32_t kNoStatus = 0xFFFFFFFFu;
static_assert(kLbBlock == 1024 && LookState::kTags == 1024, "sizes of the shared state (LookState)");

// State shared by the CTAs of a launch.
struct Shared {
  uint32_t* ticket;         // next item; zero when the launch starts
  unsigned long long* lb;   // [n_items] what the items published (Counts::word)
  unsigned long long* pre;  // [n_items / kLbBlock + 1][4] sums (look_back)
  uint32_t* late;           // [events] the launch's tag once a wait for the event's place has run out
  uint32_t* st;             // [n_items] channel statuses | bad channels << 8, where the count says so
  uint32_t tag;             // the launch's: 1 .. LookState::kTags - 1
  uint32_t n_items;         // events x FEDs
  uint32_t n_feds;
  uint32_t spin_limit;      // polls before a wait gives up
  int32_t withhold;         // failure tests: the item that never publishes its count (-1: none)
};

// Shared memory of a CTA.  TILE: digis per tile (a chunk of whole channels).
template <int TILE, bool CLUSTER>
struct __align__(16) Shm {
  // first the FED record and, per 3 bytes of it, a run slot; in the cluster kernels then
  // per digi {linking limit | kSeed, noise^2}, and at a kept cluster's first digi {its
  // last one | charge << 16, moment}
  static constexpr int kCal = CLUSTER ? TILE * (int)sizeof(uint2) : 0;
  static constexpr int kRaw = kFedBuf + kRunSlots * (int)sizeof(uint32_t);
  alignas(16) uint8_t region[((kCal > kRaw ? kCal : kRaw) + 15) / 16 * 16];
  // per digi, sorted: channel << 8 | strip (15 bits), ADC << 16, charge << 24; in the
  // cluster kernels the ADC and charge of an inactive digi are 0
  uint32_t tile[TILE];
  uint16_t list[CLUSTER ? TILE : 1];  // first digis of the seeded candidates, then of the kept ones
  int32_t mul[CLUSTER ? 2 * kCh : 1]; // the FED's charge multipliers, two per channel
  uint32_t chan_cnt[kCh + 1];         // digis before each channel
  uint32_t chan_pos[kCh];             // channel record in the FED record (or first digi in the SoA)
  uint16_t chan_len[kCh];
  uint8_t chan_st[kCh];
  unsigned long long sum64[kWarps];
  uint32_t sum[kWarps];
  uint32_t scal[4];
  __device__ __forceinline__ uint2* cal() { return reinterpret_cast<uint2*>(region); }
  __device__ __forceinline__ uint32_t* slots() { return reinterpret_cast<uint32_t*>(region + kFedBuf); }
};
constexpr uint32_t kSeed = 1u << 31;
enum { kIdx = 0, kFlags, kBad };  // scal

// The item this CTA takes, in ticket order: every item before it has then started, so
// that the waits in look_back end whatever else runs on the GPU.  meanwhile() runs
// while the ticket is on its way.  (A ticket past the last item, which only launches
// that wrongly share the state can draw: the CTA has nothing to do.)
template <class S, typename Meanwhile>
__device__ __forceinline__ uint32_t take_item(S& s, const Shared& sh, Meanwhile meanwhile) {
  uint32_t t = 0;
  if (threadIdx.x == 0) t = atomicAdd(sh.ticket, 1u);
  meanwhile();
  if (threadIdx.x == 0) s.scal[kIdx] = t;
  __syncthreads();
  return s.scal[kIdx];
}

// Sum over the CTA's threads (all call; two barriers).
template <class S>
__device__ __forceinline__ unsigned long long block_sum(S& s, unsigned long long v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  if (lane == 0) s.sum64[threadIdx.x >> 5] = v;
  __syncthreads();
  v = lane < kWarps ? s.sum64[lane] : 0ull;
#pragma unroll
  for (int d = kWarps / 2; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  v = __shfl_sync(0xffffffffu, v, 0);
  __syncthreads();
  return v;
}

// Given each warp's v (the same on all its lanes): the sum over the warps before, and
// *total over all (two barriers).
template <class S>
__device__ __forceinline__ uint32_t warps_before(S& s, uint32_t v, uint32_t* total) {
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) s.sum[warp] = v;
  __syncthreads();
  const uint32_t x = threadIdx.x % 32 < kWarps ? s.sum[threadIdx.x % 32] : 0u;
  const uint32_t pre = __reduce_add_sync(0xffffffffu, (int)(threadIdx.x % 32) < warp ? x : 0u);
  *total = __reduce_add_sync(0xffffffffu, x);
  __syncthreads();
  return pre;
}

// Exclusive prefix of v over the CTA's threads; *total their sum (two barriers).
template <class S>
__device__ __forceinline__ uint32_t block_scan(S& s, uint32_t v, uint32_t* total) {
  const int lane = threadIdx.x & 31;
  uint32_t x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  return warps_before(s, __shfl_sync(0xffffffffu, x, 31), total) + x - v;
}

// What a FED publishes in one word: clusters (at most 96 x 256), digis (the same), the
// strips of its clusters (at most 256 each), whether it has channel statuses and the
// launch's tag.  The statuses, which few FEDs have, are in a word of their own, written
// before.
struct Counts {
  uint32_t clusters = 0, digis = 0;  // (sums too: below 2^32 for SST_MAX_FEDS FEDs)
  uint32_t flags = 0, bad = 0;       // OR of the channel statuses, bad channels
  unsigned long long amps = 0;
  static constexpr unsigned long long kStatus = 1ull << 53;
  static constexpr int kTagAt = 54;
  __device__ __forceinline__ unsigned long long word(uint32_t tag) const {
    return ((unsigned long long)tag << kTagAt) | (bad ? kStatus : 0ull) | (amps << 30) |
           ((unsigned long long)digis << 15) | clusters;
  }
  __device__ __forceinline__ void add(unsigned long long w) {
    clusters += (uint32_t)w & 0x7FFFu;
    digis += (uint32_t)(w >> 15) & 0x7FFFu;
    amps += (w >> 30) & 0x7FFFFFull;
  }
};
static_assert(kCh * kStrips < 1 << 15 && kCh * kStrips * kStrips < 1 << 23 && LookState::kTags <= 1 << 10,
              "fields of a count's word");
__device__ __forceinline__ void publish(const Shared& sh, uint32_t idx, const Counts& c) {
  if (c.bad) sh.st[idx] = c.flags | (c.bad << 8);
  if ((int64_t)idx != (int64_t)sh.withhold) st_release(sh.lb + idx, c.word(sh.tag));
}

// OR over the CTA's threads (all call; two barriers).
template <class S>
__device__ __forceinline__ uint32_t block_or(S& s, uint32_t v) {
  v = __reduce_or_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) s.sum[threadIdx.x >> 5] = v;
  __syncthreads();
  v = __reduce_or_sync(0xffffffffu, threadIdx.x % 32 < kWarps ? s.sum[threadIdx.x % 32] : 0u);
  __syncthreads();
  return v;
}

// What the items lo .. idx - 1 published, summed (all threads call).  The counts of
// up to kLbBlock items are read at once, a few by each thread, so that a CTA waits for
// the slowest of them and not for a chain; further back, the last item of every
// kLbBlock publishes the sums up to and including itself, with its own counts `own`.
// STATUS: the items have statuses, wanted from item st_from on (kNoStatus: none).  A wait
// gives up after spin_limit polls: *timed_out is set and the sums are partial.
template <bool AMP, bool STATUS, class S>
__device__ __forceinline__ Counts look_back(S& s, const Shared& sh, uint32_t idx, uint32_t lo, uint32_t st_from,
                                            const Counts& own, bool* timed_out) {
  const uint32_t w0 = idx & ~(kLbBlock - 1u), from = w0 > lo ? w0 : lo;
  const bool last_of_block = lo == 0 && (idx & (kLbBlock - 1u)) == kLbBlock - 1u;
  if (last_of_block) st_from = 0;
  constexpr unsigned long long kSums = (1ull << Counts::kTagAt) - 1u;
  Counts c;
  bool to = false;
  auto poll = [&](const unsigned long long* p) -> unsigned long long {
    unsigned long long v = ld_acquire(p);
    unsigned ns = 32;
    for (uint32_t k = 0; (uint32_t)(v >> Counts::kTagAt) != sh.tag; v = ld_acquire(p)) {
      if (to || ++k > sh.spin_limit) {
        to = true;
        return 0ull;
      }
      __nanosleep(ns);
      if (ns < 256) ns <<= 1;
    }
    return v;
  };
  for (uint32_t i = from + threadIdx.x; i < idx; i += kThreads) {
    const unsigned long long w = poll(sh.lb + i);
    c.add(w);
    if (STATUS && (w & Counts::kStatus) && i >= st_from) {
      const uint32_t st = __ldcg(sh.st + i);
      c.flags |= st & 255u;
      c.bad += st >> 8;
    }
  }
  if (from > lo && threadIdx.x == 0) {  // the sums up to item from - 1
    const unsigned long long* pre = sh.pre + 4 * (size_t)(from / kLbBlock - 1);
    c.clusters += (uint32_t)(poll(pre) & kSums);
    if (!to) {
      c.digis += (uint32_t)__ldcg(pre + 1);
      c.amps += __ldcg(pre + 2);
      if (STATUS && st_from != kNoStatus) {
        const unsigned long long st = __ldcg(pre + 3);
        c.flags |= (uint32_t)(st >> 32);
        c.bad += (uint32_t)st;
      }
    }
  }
  // clusters and digis in one sum (each below 2^32 within one block of items)
  if (w0 <= lo && !AMP) {
    const unsigned long long both = block_sum(s, c.clusters | ((unsigned long long)c.digis << 32));
    c.clusters = (uint32_t)both;
    c.digis = (uint32_t)(both >> 32);
  } else {
    c.clusters = (uint32_t)block_sum(s, c.clusters);
    c.digis = (uint32_t)block_sum(s, c.digis);
    if (AMP) c.amps = block_sum(s, c.amps);
  }
  if (STATUS && st_from != kNoStatus && __syncthreads_or(c.bad != 0)) {
    c.flags = block_or(s, c.flags);
    c.bad = (uint32_t)block_sum(s, c.bad);
  }
  to = __syncthreads_or(to);
  if (threadIdx.x == 0 && last_of_block && (int64_t)idx != (int64_t)sh.withhold) {
    unsigned long long* pre = sh.pre + 4 * (size_t)(idx / kLbBlock);
    pre[1] = c.digis + own.digis;
    pre[2] = c.amps + own.amps;
    pre[3] = ((unsigned long long)(c.flags | own.flags) << 32) | (c.bad + own.bad);
    __threadfence();
    st_release(pre, ((unsigned long long)sh.tag << Counts::kTagAt) | (c.clusters + own.clusters));
  }
  *timed_out = to;
  return c;
}

// An event's flags, written by its last FED's CTA (which has seen every FED's count,
// and with it the statuses), and SST_EV_TIMEOUT when a wait for the event's place ran
// out.  A CTA whose wait did marks the event's word and then adds the flag; with the word
// read after the flags are written, one of the two is seen.
__device__ __forceinline__ void write_flags(const Shared& sh, uint32_t e, uint32_t flags, sst_event_status* st) {
  volatile uint32_t* f = &st->flags;
  *f = flags;
  __threadfence();
  if (atomicOr(sh.late + e, 0u) == sh.tag) atomicOr(&st->flags, SST_EV_TIMEOUT);
}
__device__ __forceinline__ void flag_timeout(const Shared& sh, uint32_t e, sst_event_status* st) {
  atomicExch(sh.late + e, sh.tag);
  __threadfence();
  atomicOr(&st->flags, SST_EV_TIMEOUT);
}

// ---------------------------------------------------------------- FED record (a1, a2)

// An event's FED lengths, loaded before the CTA knows its FED.
struct Lengths {
  static constexpr int kN = 2;
  uint32_t v[kN];
  __device__ __forceinline__ void load(const uint32_t* __restrict__ len_e, uint32_t n_feds) {
#pragma unroll
    for (int u = 0; u < kN; u++) {
      const uint32_t i = threadIdx.x + u * kThreads;
      v[u] = i < n_feds ? __ldg(len_e + i) : 0u;
    }
  }
};

// Byte offset of FED f's record (all threads call): the event's start ev0 plus the
// lengths before it; *len its own, *ok whether it ends within the event (by ev1),
// *size_ok (of the last FED) whether the lengths add up to the event's bytes.
template <class S>
__device__ __forceinline__ uint64_t find_fed(S& s, const Lengths& first, const uint32_t* __restrict__ len_e,
                                             uint32_t f, uint32_t n_feds, uint64_t ev0, uint64_t ev1, uint32_t* len,
                                             bool* ok, bool* size_ok) {
  const uint32_t l = __ldg(len_e + f);
  unsigned long long part = 0;
#pragma unroll
  for (int u = 0; u < Lengths::kN; u++)
    if (threadIdx.x + u * kThreads < f) part += first.v[u];
  for (uint32_t i = threadIdx.x + Lengths::kN * kThreads; i < f; i += kThreads) part += __ldg(len_e + i);
  const uint64_t o = ev0 + block_sum(s, part);
  *ok = ev1 >= ev0 && o + l <= ev1;
  *size_ok = f + 1 < n_feds || o + l == ev1;
  *len = *ok ? l : 0u;
  return o;
}

// Stages the record when it fits the region (19 KB; beyond kFedBuf the run slots' space
// holds the rest); returns where its bytes are.
template <class S>
__device__ __forceinline__ const uint8_t* stage_record(S& s, const uint8_t* g, uint32_t len) {
  if (len == 0 || len > (uint32_t)sizeof(s.region)) return g;
  if ((reinterpret_cast<uintptr_t>(g) & 15u) == 0) {
    const uint32_t nv = len >> 4;
    for (uint32_t i = threadIdx.x; i < nv; i += kThreads)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(s.region + 16 * i)),
                   "l"(g + 16 * i)
                   : "memory");
    for (uint32_t i = (nv << 4) + threadIdx.x; i < len; i += kThreads) s.region[i] = __ldg(g + i);
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else {
    for (uint32_t i = threadIdx.x; i < len; i += kThreads) s.region[i] = __ldg(g + i);
  }
  __syncthreads();
  return s.region;
}

// Validates one channel record's runs in order (rd reads its bytes) and counts its
// digis; the first error found decides the status.  note(p, digis before) sees every
// valid run's header.
template <typename Rd, typename Note>
__device__ __forceinline__ uint32_t count_runs(uint32_t len, Rd rd, uint32_t* st, Note note) {
  if (rd(2) != SST_ZS_CODE) {
    *st = SST_CH_BAD_CODE;
    return 0;
  }
  uint32_t p = 3, prev_end = 0, cnt = 0;
  while (p + 2 <= len) {
    const uint32_t f = rd(p), wd = rd(p + 1), np = p + 2 + wd;
    const bool range = wd - 1u > (uint32_t)kStrips - 1u - f;  // width 0, or past strip 256
    if (range || f < prev_end || np > len) {
      *st = range ? SST_CH_RUN_RANGE : f < prev_end ? SST_CH_RUN_ORDER : SST_CH_TRUNC;
      return 0;
    }
    note(p, cnt);
    prev_end = f + wd;
    cnt += wd;
    p = np;
  }
  if (p != len) {  // a header cut by the record end
    *st = SST_CH_TRUNC;
    return 0;
  }
  return cnt;
}

// Thread per channel: cnt digis of channel tid (threads past the last: 0) to chan_cnt;
// the channel statuses to scal[kFlags], scal[kBad]; returns all digis.  Barriers on
// the way and at the end.
template <class S>
__device__ __forceinline__ uint32_t prefix_counts(S& s, uint32_t cnt) {
  const int tid = threadIdx.x;
  uint32_t total;
  const uint32_t pre = block_scan(s, cnt, &total);
  if (tid < kCh) s.chan_cnt[tid] = pre;
  if (tid == 0) s.chan_cnt[kCh] = total;
  if (tid < 32) {
    uint32_t fl = 0, nb = 0;
    for (int c = tid; c < kCh; c += 32) {
      fl |= s.chan_st[c];
      nb += s.chan_st[c] ? 1u : 0u;
    }
    fl = __reduce_or_sync(0xffffffffu, fl);
    nb = __reduce_add_sync(0xffffffffu, nb);
    if (tid == 0) {
      s.scal[kFlags] = fl;
      s.scal[kBad] = nb;
    }
  }
  __syncthreads();
  return total;
}

// FED header, channel length chains, run validation and digi counts.  src: the
// record's bytes (shared or global).  On return chan_* describe every channel,
// chan_cnt the digis before it (chan_cnt[96]: all), scal[kFlags] / scal[kBad] the OR
// of the channel statuses and the number of bad channels.  SLOTS (src is the staged
// record, of at most kFedBuf bytes): every valid run's header position | digis of the channel before it << 13 |
// channel << 21 | 1 << 31 is left in the slot of its position / 3 (headers are at least
// 3 bytes apart); the channels are as good as their statuses say.  Returns the digis.
template <bool SLOTS, class S>
__device__ __forceinline__ uint32_t parse_record(S& s, const uint8_t* src, uint32_t len, uint32_t fed, bool in_range) {
  static_assert(kFedBuf <= 1 << 13, "header positions take 13 bits of a slot");
  const int tid = threadIdx.x, lane = tid & 31;
  if (SLOTS)
    for (uint32_t i = tid; i < (len + 2) / 3; i += kThreads) s.slots()[i] = 0;
  if (tid < 32) {
    // header: lanes 0 .. 7 hold one FE unit each
    const bool present = in_range && len > 0;
    bool ok = present && len >= (uint32_t)kHdr;
    uint32_t fl = 0, start = 0;
    if (ok) {
      fl = lane < kFe ? rd16(src + 16 + 2 * lane) : 0u;
      const uint32_t padded = (fl + 7u) & ~7u;
      uint32_t x = padded;
#pragma unroll
      for (int d = 1; d < 8; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
      }
      start = kHdr + x - padded;
      const uint32_t total = (kHdr + __shfl_sync(0xffffffffu, x, kFe - 1) + 15u) & ~15u;
      bool hdr = true;
      if (lane == 0)
        hdr = rd32(src) == SST_FED_MAGIC && rd16(src + 4) == fed && src[6] == (uint8_t)kCh &&
              src[7] == (uint8_t)kFe && rd32(src + 8) == len && total == len;
      ok = __shfl_sync(0xffffffffu, hdr, 0);
    }
    if (lane < kFe) {
      bool good = false;
      if (ok)
        good = cs::walk_lengths(start, fl, [&](uint32_t i) { return (uint32_t)src[i]; },
                                [&](int k, uint32_t pos, uint32_t l) {
                                  s.chan_pos[lane * kChPerFe + k] = pos;
                                  s.chan_len[lane * kChPerFe + k] = (uint16_t)l;
                                });
      const uint8_t st = good ? 0 : ok ? (uint8_t)SST_CH_FRAMING
                                  : !in_range || present ? (uint8_t)SST_CH_FED_HDR : (uint8_t)0;
#pragma unroll
      for (int k = 0; k < kChPerFe; k++) {
        const int c = lane * kChPerFe + k;
        if (!good) s.chan_pos[c] = s.chan_len[c] = 0;
        s.chan_st[c] = st;
      }
    }
  }
  __syncthreads();
  uint32_t cnt = 0, st = 0;
  if (tid < kCh) {
    st = s.chan_st[tid];
    const uint32_t l = s.chan_len[tid];
    if (st == 0 && l >= 3) {
      const uint32_t pos = s.chan_pos[tid];
      const uint8_t* r = src + pos;
      cnt = count_runs(l, [&](uint32_t i) { return (uint32_t)r[i]; }, &st, [&](uint32_t p, uint32_t before) {
        if (SLOTS) s.slots()[(pos + p) / 3] = (pos + p) | (before << 13) | ((uint32_t)tid << 21) | (1u << 31);
      });
      s.chan_st[tid] = (uint8_t)st;
    }
  }
  return prefix_counts(s, cnt);
}

// Greedy chunk of whole channels [c0, result) with at most TILE digis.
template <int TILE, class S>
__device__ __forceinline__ int chunk_end(const S& s, int c0) {
  int c1 = c0 + 1;
  while (c1 < kCh && s.chan_cnt[c1 + 1] - s.chan_cnt[c0] <= (uint32_t)TILE) ++c1;
  return c1;
}

// Copies the runs of channels [c0, c1) into the tile: groups of `lanes` threads share
// a channel, all walk its run headers, each copies every lanes-th ADC byte.  Records
// were validated; the copy is still bounded by the counted digis so that it cannot
// leave the tile.  Ends with a barrier.
template <class S>
__device__ __forceinline__ void emit_channels(S& s, const uint8_t* src, int c0, int c1, int lanes) {
  const int gid = threadIdx.x / lanes, li = threadIdx.x % lanes, ng = kThreads / lanes;
  const uint32_t base = s.chan_cnt[c0];
  for (int c = c0 + gid; c < c1; c += ng) {
    const uint32_t o0 = s.chan_cnt[c] - base;
    const uint32_t n = s.chan_cnt[c + 1] - s.chan_cnt[c];
    if (n == 0) continue;
    const uint8_t* r = src + s.chan_pos[c];
    const uint32_t len_c = s.chan_len[c];
    uint32_t p = 3, o = 0;
    while (p + 2 <= len_c && o < n) {
      const uint32_t first = r[p];
      uint32_t w = r[p + 1];
      p += 2;
      if (w > n - o) w = n - o;
      for (uint32_t k = li; k < w; k += lanes)
        s.tile[o0 + o + k] = ((uint32_t)c << 8) | ((first + k) & 255u) | ((uint32_t)r[p + k] << 16);
      o += w;
      p += w;
    }
  }
  __syncthreads();
}

// The same for all channels of a record with run slots, a thread each.
template <class S>
__device__ __forceinline__ void emit_slots(S& s, uint32_t len) {
  for (uint32_t i = threadIdx.x; i < (len + 2) / 3; i += kThreads) {
    const uint32_t d = s.slots()[i];
    if (!d) continue;
    const uint32_t c = (d >> 21) & 127u;
    if (s.chan_st[c]) continue;  // a corrupt channel: no digis
    const uint8_t* r = s.region + (d & 0x1FFFu);
    const uint32_t first = r[0], w = r[1], o = s.chan_cnt[c] + ((d >> 13) & 255u);
    for (uint32_t k = 0; k < w; k++)
      s.tile[o + k] = (c << 8) | (first + k) | ((uint32_t)r[2 + k] << 16);
  }
  __syncthreads();
}

// ---------------------------------------------------------------- clustering (a3 - a6)

// a3 of one digi of the tile: its calibration entry v decides whether it is active and
// a seed; tile and cal receive what the later steps read.
template <class S>
__device__ __forceinline__ void classify(S& s, uint32_t i, uint32_t key, uint32_t adc, uint2 v) {
  const bool act = adc > (v.x & 255u), seed = adc > ((v.x >> 8) & 255u);
  uint32_t t = key;
  if (act) t |= (adc << 16) | (cs::charge(adc, s.mul[key >> 7]) << 24);
  s.tile[i] = t;
  s.cal()[i] = make_uint2((v.x >> 16) | (seed ? kSeed : 0u), v.y);
}
constexpr uint32_t kNeverActive = 0xFFFFu;  // a calibration word with both limits 255

// Classifies the n digis that are in the tile.  Ends with a barrier.
template <class S>
__device__ __forceinline__ void classify_tile(S& s, const uint2* __restrict__ cal0, uint32_t n) {
  constexpr int kU = 4;  // gathers in flight per thread
  for (uint32_t i0 = threadIdx.x; i0 < n; i0 += kU * kThreads) {
    uint2 v[kU];
    uint32_t t[kU];
#pragma unroll
    for (int u = 0; u < kU; u++) {
      const uint32_t i = i0 + u * kThreads;
      t[u] = i < n ? s.tile[i] : 0u;
      v[u] = __ldg(cal0 + (t[u] & 0x7FFFu));
    }
#pragma unroll
    for (int u = 0; u < kU; u++)
      if (i0 + u * kThreads < n) classify(s, i0 + u * kThreads, t[u] & 0x7FFFu, (t[u] >> 16) & 255u, v[u]);
  }
  __syncthreads();
}

// The active digi before digi i in its channel that i is linked to, or -1: i starts a
// candidate (cs::walk_any has the rule).  Nearly every recorded strip is active, so the
// search is a step or two.
template <class S>
__device__ __forceinline__ int linked_before(S& s, int i) {
  const uint32_t k = s.tile[i] & 0x7FFFu;
  int j = i - 1;
  uint32_t t = 0;
  while (j >= 0 && !((t = s.tile[j]) >> 16) && (t >> 8) == (k >> 8)) --j;
  if (j < 0 || ((t & 0x7FFFu) >> 8) != (k >> 8)) return -1;
  return (k & 255u) - (t & 255u) - 1u < (s.cal()[i].x & 255u) ? j : -1;
}

// Finds the kept clusters among the tile's n classified digis; lists their first digis
// in order and returns how many.  A kept cluster's first digi's cal entry becomes {last
// active digi | charge << 16, moment (of strip x charge)}.
//  1. a thread per digi: a seed walks back to its candidate's start and stands for it
//     unless it meets another seed; the starts are listed in order;
//  2. a thread per listed candidate: the sums in strip order (3 digis on average),
//     the cluster threshold; the kept ones move up in the list.
// One lane per channel (the walk of k_stream) is the cheaper way with many events in
// flight; here its 30 dependent steps were the kernel's critical path.  Ends with a
// barrier.
template <int TILE, class S>
__device__ __forceinline__ uint32_t find_clusters(S& s, uint32_t n, float t_cluster) {
  constexpr int kStretch = (TILE + kThreads - 1) / kThreads;  // windows of a warp
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t part = (n + kThreads - 1) / kThreads * 32;
  const uint32_t b0 = warp * part, b1 = b0 + part < n ? b0 + part : n;
  int own[kStretch];
  uint32_t cnt = 0, n_cand;
#pragma unroll
  for (int k = 0; k < kStretch; k++) {
    own[k] = -1;
    const uint32_t i = b0 + 32 * k + lane;
    if (b0 + 32 * k < b1) {
      if (i < b1 && (s.cal()[i].x & kSeed)) {
        int j = (int)i;
        for (;;) {
          const int p = linked_before(s, j);
          if (p < 0) {
            own[k] = j;
            break;
          }
          if (s.cal()[p].x & kSeed) break;
          j = p;
        }
      }
      cnt += __popc(__ballot_sync(0xffffffffu, own[k] >= 0));
    }
  }
  uint32_t o = warps_before(s, cnt, &n_cand);
#pragma unroll
  for (int k = 0; k < kStretch; k++)
    if (b0 + 32 * k < b1) {
      const unsigned m = __ballot_sync(0xffffffffu, own[k] >= 0);
      if (own[k] >= 0) s.list[o + __popc(m & ((1u << lane) - 1u))] = (uint16_t)own[k];
      o += __popc(m);
    }
  __syncthreads();
  const cs::Threshold thr(t_cluster);
  uint32_t kept = 0;
  for (uint32_t r0 = 0; r0 < n_cand; r0 += kThreads) {
    const bool have = r0 + threadIdx.x < n_cand;
    bool pass = false;
    uint32_t i = 0, sums = 0, moment = 0, last = 0;
    if (have) {
      last = i = s.list[r0 + threadIdx.x];
      uint32_t t = s.tile[i];
      const uint32_t c = t >> 8 & 127u;
      uint2 v = s.cal()[i];
      float n2 = 0.f;
      for (uint32_t j = i;;) {
        const uint32_t q = t >> 24, a = (t >> 16) & 255u, st = t & 255u;
        if (a) {
          sums += (q << 16) + a;
          moment += st * q;
          n2 = __fadd_rn(n2, __uint_as_float(v.y));
          last = j;
        }
        if (++j >= n) break;
        t = s.tile[j];
        v = s.cal()[j];
        if (((t >> 8) & 127u) != c) break;
        if ((t >> 16) && (t & 255u) - (s.tile[last] & 255u) - 1u >= (v.x & 255u)) break;  // the next candidate
      }
      pass = thr.pass(sums & 0xFFFFu, n2);
    }
    const unsigned m = __ballot_sync(0xffffffffu, pass);
    uint32_t all;
    const uint32_t at = kept + warps_before(s, __popc(m), &all) + __popc(m & ((1u << lane) - 1u));
    // (behind the barriers: the candidate before this one has looked at cal()[i], its end)
    if (pass) {
      s.cal()[i] = make_uint2(last | (sums & 0xFFFF0000u), moment);
      s.list[at] = (uint16_t)i;  // at or before the place it was read from
    }
    kept += all;
    __syncthreads();
  }
  return kept;
}

// A kept cluster's strips [lo, hi] of channel c, widened over up to max_adj adjacent
// bad strips at either end; i: its first digi.
template <class S>
__device__ __forceinline__ void cluster_strips(S& s, const KParams& kp, uint32_t fed, uint32_t i, int* lo, int* hi,
                                               uint32_t* c) {
  const uint32_t k = s.tile[i] & 0x7FFFu;
  *c = k >> 8;
  *lo = (int)(k & 255u);
  *hi = (int)(s.tile[s.cal()[i].x & 0xFFFFu] & 255u);
  if (kp.max_adj > 0) {
    const uint32_t* m = kp.badmask + ((size_t)fed * kCh + *c) * kMaskWords;
    for (int j = 0; j < kp.max_adj && *lo > 0 && bit(m, *lo - 1); j++) --*lo;
    for (int j = 0; j < kp.max_adj && *hi + 1 < kStrips && bit(m, *hi + 1); j++) ++*hi;
  }
}

// Where an event's clusters go.
struct Out {
  uint64_t off, room;          // its slice of the SoA
  uint64_t a_off = 0, a_room = 0;  // and of the amplitudes
};

// Threads to a channel that leave none idle in a chunk of n channels.
__device__ __forceinline__ int lanes_for(int n) {
  int l = 32;
  while (l > 2 && l * n > kThreads) l /= 2;
  return l;
}

// Clusters one FED whose `total` digis load(c0, c1) brings into the tile, classified,
// chunk by chunk, and writes its clusters in order.  A FED of more than one chunk leaves
// its clusters in `spill` (kFedClusters of them) until it knows their place; with
// amplitudes, without a spill area, or with more clusters (digis given in no order may
// each be one), it goes through the chunks again (17 events of 13 FEDs of very different
// density, from host memory: 863 us twice, 406 once).
// place(found, amps) publishes the counts and returns those of the FEDs before.  Returns
// the clusters found; *amps_found their strips.
template <bool AMP, int TILE, class S, typename Load, typename Place>
__device__ __forceinline__ uint32_t cluster_fed(S& s, const KParams& kp, uint32_t fed, uint32_t total, Load load,
                                                Place place, const Out& o, const sst_clusters& out, uint2* spill,
                                                uint32_t* amps_found) {
  const bool single = total <= (uint32_t)TILE;
  uint32_t in_tile = 0;  // kept clusters of the chunk in the tile
  auto chunk = [&](int c0, int c1) {
    const uint32_t n = s.chan_cnt[c1] - s.chan_cnt[c0];
    in_tile = 0;
    if (n == 0) return;
    load(c0, c1);
    in_tile = find_clusters<TILE>(s, n, kp.t_cluster);
  };
  uint32_t found = 0, amps = 0;
  for (int c0 = 0; c0 < kCh;) {
    const int c1 = single ? kCh : chunk_end<TILE>(s, c0);
    chunk(c0, c1);
    if (!AMP && !single && spill)
      for (uint32_t r = threadIdx.x; r < in_tile && found + r < kFedClusters; r += kThreads) {
        int lo, hi;
        uint32_t c;
        const uint32_t i = s.list[r];
        cluster_strips(s, kp, fed, i, &lo, &hi, &c);
        const uint2 v = s.cal()[i];
        spill[found + r] =
            cs::staged_cluster((uint32_t)lo, (uint32_t)(hi - lo + 1), v.x >> 16, v.y - (uint32_t)lo * (v.x >> 16), c);
      }
    if (!single) __syncthreads();  // the tile is filled again
    found += in_tile;
    if (AMP) {
      uint32_t w = 0;
      for (uint32_t r = threadIdx.x; r < in_tile; r += kThreads) {
        int lo, hi;
        uint32_t c;
        cluster_strips(s, kp, fed, s.list[r], &lo, &hi, &c);
        w += (uint32_t)(hi - lo + 1);
      }
      amps += (uint32_t)block_sum(s, w);
    }
    c0 = c1;
  }
  const Counts before = place(found, amps);
  const unsigned long long n0 = before.clusters, a0 = before.amps;
  *amps_found = amps;
  if (!AMP && !single && spill && found <= kFedClusters) {
    for (uint32_t r = threadIdx.x; r < found && n0 + r < o.room; r += kThreads) {
      const uint2 v = spill[r];
      const uint32_t lo = v.x & 255u, wd = ((v.x >> 8) & 255u) + 1u, q = v.x >> 16;
      const uint64_t at = o.off + n0 + r;
      out.det[at] = fed * (uint32_t)kCh + (v.y >> 24);
      out.first[at] = (uint16_t)lo;
      out.width[at] = (uint16_t)wd;
      out.charge[at] = q;
      out.barycenter[at] = centroid(lo, wd, q, v.y & 0xFFFFFFu);
    }
    return found;
  }
  uint32_t run = 0, arun = 0;  // clusters and strips of the chunks before
  for (int c0 = 0; c0 < kCh && found > 0;) {
    const int c1 = single ? kCh : chunk_end<TILE>(s, c0);
    if (!single) {
      __syncthreads();  // the tile is filled again
      chunk(c0, c1);
    }
    for (uint32_t r0 = 0; r0 < in_tile; r0 += kThreads) {
      const uint32_t r = r0 + threadIdx.x;
      const bool have = r < in_tile;
      int lo = 0, hi = -1;
      uint32_t c = 0, i = 0;
      if (have) {
        i = s.list[r];
        cluster_strips(s, kp, fed, i, &lo, &hi, &c);
      }
      const uint32_t wd = (uint32_t)(hi - lo + 1);
      uint32_t a_at = 0, a_tot = 0;
      bool amp_fits = false;
      if (AMP) {
        a_at = block_scan(s, wd, &a_tot);
        amp_fits = a0 + arun + a_at + wd <= o.a_room;
        if (have && amp_fits) {
          uint8_t* d = out.amp + o.a_off + a0 + arun + a_at;
          for (uint32_t k = 0; k < wd; k++) d[k] = 0;
          const uint32_t last = s.cal()[i].x & 0xFFFFu;
          for (uint32_t j = i; j <= last; j++) {
            const uint32_t t = s.tile[j];
            if (t >> 16) d[(int)(t & 255u) - lo] = (uint8_t)(t >> 24);  // active
          }
        }
      }
      if (have && n0 + run + r < o.room) {
        const uint2 v = s.cal()[i];
        const uint32_t q = v.x >> 16;
        const uint64_t at = o.off + n0 + run + r;
        out.det[at] = fed * (uint32_t)kCh + c;
        out.first[at] = (uint16_t)lo;
        out.width[at] = (uint16_t)wd;
        out.charge[at] = q;
        out.barycenter[at] = centroid((uint32_t)lo, wd, q, v.y - (uint32_t)lo * q);
        if (AMP) out.amp_first[at] = amp_fits ? (uint32_t)(o.a_off + a0 + arun + a_at) : kNoAmp;
      }
      arun += a_tot;
    }
    run += in_tile;
    c0 = c1;
  }
  return found;
}

}  // namespace ev

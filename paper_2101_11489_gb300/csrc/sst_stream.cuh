// sst_stream.cuh -- channel streams: unpacking and clustering with one lane per
// channel record (arXiv 2101.11489, section 2: channels are independent of one
// another, clusters never cross a channel).
//
// A lane reads its channel's bytes once, front to back, and carries everything the
// method needs in registers: the run it is in, the open candidate's sums (raw ADC,
// noise^2, gain-corrected charge, first moment), its first and last active strip and
// whether it has a seed.  Unpacking, thresholds, the candidate rule and the sums of
// one digi are one step of that walk; no digi is stored.  When an active strip is
// not linked to the one before it, the open candidate ends; a seeded one leaves a
// 16-byte record in the warp's list.  The list is then finished with one lane per
// record: cluster threshold, place in the output.
//
// Included by sst_kernels.cu only, inside its namespace.
#pragma once

namespace cs {

constexpr uint32_t kNotKept = 0xFFFFFFFFu;
constexpr int kRefill = 12;  // lanes still walking when the others take new channels
// Dynamic shared memory of a CTA whose shared addresses fit the 16 bits that Walk::from has
// for them (2 KB are left to static variables and the system).
constexpr size_t kFromLimit = 65536 - 2048;

// Per-warp shared memory.  A warp takes up to 4 U slots at once, a slot being C = 12
// (or 6) consecutive channels of one FE unit of one event.  With U = 2 eight warps
// and a tile of calibration entries fit four times on an SM.
template <int U>
struct __align__(16) WarpT {
  static constexpr int kSlots = 4 * U;
  static constexpr int kTasks = kSlots * kChPerFe;   // channels, one lane each
  static constexpr int kBuf = U == 2 ? 3216 : 1616;  // bytes of FE units staged
  static constexpr uint32_t kMaxRec = kBuf / 2 > 1536 ? kBuf / 2 : 1536;  // most candidates at once (List)
  struct Slot {
    uint32_t room[kSlots];   // staging records of the slot's event
    uint32_t digis[kSlots], flags[kSlots], nbad[kSlots];  // digis, OR of channel statuses, bad channels
  };
  uint8_t buf[kBuf];         // the FE units' bytes, each unit at a multiple of 8 (the walk may read 2 past the last)
  uint64_t base[kSlots];     // first staging record of the slot's event
  uint32_t task[kTasks];     // byte position | length << 16 of every channel record; after the walk, the
                             // place of the channel's first kept cluster in its event's staging slice
  union {
    Slot slot;
    uint32_t bins[32];       // the ordering's counts, before
  };
  uint8_t kept[kTasks];      // kept clusters per channel (at most 128)
  uint8_t order[kTasks];     // channels, longest record first
};
template <int U>
constexpr bool layout_ok() {
  using W = WarpT<U>;
  return offsetof(W, base) % 8 == 0 && sizeof(W) % 16 == 0 && W::kBuf % 16 == 0 && W::kTasks <= 128 &&
         W::kMaxRec <= kSpillRecords;
}
static_assert(layout_ok<1>() && layout_ok<2>(), "per-warp shared memory layout");

// The warp's candidate list, in its spill area in global memory (in L2: the areas
// are used over and over).  A channel record of n bytes has at most n / 2
// candidates (consecutive ones start at least two bytes apart) and at most 128
// (their strips ascend), so neither a full staging buffer nor one FE unit read in
// place has more than kMaxRec.  On chip, 2 KB of records per warp cost the fourth
// CTA of an SM: 226 against 185 us (64 full-detector events).
// Record: {first strip | last + 1 << 8 | task << 17; raw ADC | charge << 16;
// noise^2, then place among the task's kept clusters; moment}.
// Clusters with amplitudes: `from` says where a record's first digi is (Walk::from); 128
// words after its kSpillRecords are free for per-task values.
struct List {
  uint4* rec;
  uint32_t* from;
  uint32_t n;
  // Appends r of every lane with `emit` (all lanes call).
  template <bool AMP>
  __device__ __forceinline__ void append(bool emit, uint4 r, uint32_t at) {
    const unsigned b = __ballot_sync(0xffffffffu, emit);
    const uint32_t i = n + __popc(b & ((1u << (threadIdx.x & 31)) - 1u));
    if (emit && i < kSpillRecords) {
      rec[i] = r;
      if (AMP) from[i] = at;
    }
    n += __popc(b);
  }
};

// The cluster threshold: a cluster is kept when its raw charge s is larger than the
// binary32 product t x sqrt(n2).  s^2 and t^2 n2 decide that whenever they differ by
// more than four parts in a million (the roundings of either form stay below 2^-21
// relative); the rest, and thresholds whose square leaves the normal range, take the
// product.
struct Threshold {
  float t, t2, margin;
  __device__ __forceinline__ explicit Threshold(float t_cluster) {
    t = t_cluster;
    t2 = __fmul_rn(t, t);
    margin = t2 > 1e-20f && t2 < 1e20f ? 4e-6f : __int_as_float(0x7f800000);
  }
  __device__ __forceinline__ bool pass(uint32_t charge, float n2) const {
    const float s = __uint2float_rn(charge), a = __fmul_rn(s, s), b = __fmul_rn(t2, n2);
    bool p = a > b;
    if (!(fabsf(__fsub_rn(a, b)) > __fmul_rn(margin, b))) p = s > __fmul_rn(t, __fsqrt_rn(n2));
    return p;
  }
};

// Gain-corrected charge (section 2): the ADC times the APV's certified fixed-point
// multiplier m, half up (k_gain_pack); for the rare APV without one, m negative, the
// bits of -gain: the quotient itself.  Capped at 254; saturation codes are kept.
__device__ __forceinline__ uint32_t charge(uint32_t adc, int32_t m) {
  uint32_t q = (adc * (uint32_t)m + (1u << (kMulShift - 1))) >> kMulShift;
  if (m < 0) {
    const float y = __fadd_rn(__fdiv_rn(__uint2float_rn(adc), -__int_as_float(m)), 0.5f);
    q = y >= 254.f ? 254u : (uint32_t)y;
  }
  return adc >= 254u ? adc : (q < 254u ? q : 254u);
}

// A lane's place in its channel record and its open candidate.
struct Walk {
  uint32_t p;          // next byte
  uint32_t strip;      // next strip
  uint32_t strip_end;  // strip past the run; strip == strip_end: a run header comes next
  uint32_t first;      // the candidate's first strip | task << 17
  uint32_t last1;      // its last active strip + 1
  uint32_t sums;       // raw ADC | charge << 16
  uint32_t moment;     // sum of strip x charge
  float n2;            // sum of noise^2, strip by strip
  uint32_t seeded;     // it has a seed
  uint32_t digis;      // digis read
  uint32_t from;       // amplitudes: byte after the candidate's first digi (16 bits) | strip past its run << 16
  __device__ __forceinline__ void begin(uint32_t pos) {
    p = pos;
    strip = strip_end = from = 0;
    first = sums = moment = seeded = digis = 0;
    last1 = 0u - 4096u;  // the first active strip starts a candidate, whatever its linking limit
    n2 = 0.f;
  }
  __device__ __forceinline__ uint4 record() const {
    return make_uint4(first + (last1 << 8), sums, __float_as_uint(n2), moment);
  }
};

// The walk itself, for channel records staged in shared memory and APVs that all
// have a certified multiplier.  Every step takes one digi of every lane still
// walking; a lane at a run header reads the header and the run's first digi in one
// step.  A lane stops (p stays) at its record's end or at a header that breaks a
// rule: width 0, past strip 256, before the end of the run before it, or past the
// record's end; all four fold into one predicate.  Returns when at most `few` lanes
// are walking, with whether this one is.
//
// The step is straight-line predicated code, written as PTX because the compiler's
// own version of the same step branches around its parts (88 instructions a step
// against about 65, 12 of them only when some lane ends a seeded candidate).  A digi is
// fetched (header, ADC, calibration entry) one step before it is used, so that the
// loads' latency is covered by the step between; on return the digi fetched last is
// given back.  How many lanes still walk is looked at every second step.
//   end2  the record's end - 2 (0: the lane has no record);  cal: its channel's
//   calibration entries (DIRECT: in global memory, else shared);  m0, m1: its APVs'
//   multipliers;  task17: its task << 17;  list.n: on return with the records appended.

// Fetches the next digi of a lane that was (WAS) and is (AL) still walking: strip S, ADC A, calibration
// entry {C, N}.  A run header, when one comes next, is `ok` when its bytes end within the
// record, its strips within the channel, its width is not 0 and it starts after the run
// before it.
  #define CS_FETCH(S, A, C, N, F, AL, WAS, END2, ENTRY, ON_FETCH) \
  "setp.eq.and.u32 hdr, %1, %2, " WAS ";\n" \
  "@hdr ld.shared.u8 b0, [%0];\n" \
  "@hdr ld.shared.u8 b1, [%0+1];\n" \
  "add.u32 e, %0, b1;\n" \
  "add.u32 u, b0, b1;\n" \
  "setp.le.and.u32 ok, e, %" END2 ", hdr;\n" \
  "setp.le.and.u32 ok, u, 256, ok;\n" \
  "setp.lt.and.u32 ok, b0, u, ok;\n" \
  "setp.ge.and.u32 ok, b0, %1, ok;\n" \
  "not.pred " AL ", hdr;\n" \
  "and.pred " AL ", " AL ", " WAS ";\n" \
  "or.pred " AL ", " AL ", ok;\n" \
  "@ok mov.u32 %1, b0;\n" \
  "@ok mov.u32 %2, u;\n" \
  "@ok add.u32 %0, %0, 2;\n" \
  "mov.u32 " S ", %1;\n" \
  "@" AL " ld.shared.u8 " A ", [%0];\n" \
  ENTRY(S, C, N, AL) \
  "@" AL " add.u32 %0, %0, 1;\n" \
  "@" AL " add.u32 %1, " S ", 1;\n" \
  ON_FETCH(F)
// Uses a fetched digi: whether it is active, a seed, not linked to the active strip before
// it; the seeded candidates that end here go to the list; the gain-corrected charge (adc
// x multiplier, half up, capped at 254, saturation codes kept); the open candidate.
// Operands 0 - 11 are the walk's state, the arguments the numbers of the others;
// ON_FETCH, ON_EMIT and ON_START add what clusters with amplitudes need.
  #define CS_USE(S, A, C, N, F, AL, NEXT, M0, M1, LT, REC, HALF, SHIFT, T17, ON_EMIT, ON_START) \
  "@" AL " add.u32 %9, %9, 1;\n" \
  "and.b32 lo, " C ", 255;\n" \
  "setp.gt.and.u32 act, " A ", lo, " AL ";\n" \
  "bfe.u32 hi, " C ", 8, 8;\n" \
  "setp.gt.and.u32 seed, " A ", hi, act;\n" \
  "shr.u32 gap, " C ", 16;\n" \
  "sub.u32 d, " S ", %4;\n" \
  "setp.ge.and.u32 start, d, gap, act;\n" \
  "and.pred emit, start, seeded;\n" \
  "vote.sync.ballot.b32 bal, emit, 0xffffffff;\n" \
  "setp.eq.u32 t, bal, 0;\n" \
  "@t bra.uni " NEXT ";\n" \
  "and.b32 i, bal, %" LT ";\n" \
  "popc.b32 i, i;\n" \
  "add.u32 i, i, %10;\n" \
  "popc.b32 d, bal;\n" \
  "add.u32 %10, %10, d;\n" \
  "mad.lo.u32 x, %4, 256, %3;\n" \
  "mov.b32 d, %7;\n" \
  "mad.wide.u32 g, i, 16, %" REC ";\n" \
  "@emit st.global.v4.u32 [g], {x, %5, d, %6};\n" \
  ON_EMIT \
  NEXT ":\n" \
  "setp.lt.u32 t, " S ", 128;\n" \
  "selp.u32 m, %" M0 ", %" M1 ", t;\n" \
  "mad.lo.u32 q, " A ", m, %" HALF ";\n" \
  "shr.u32 q, q, %" SHIFT ";\n" \
  "min.u32 q, q, 254;\n" \
  "setp.ge.u32 t, " A ", 254;\n" \
  "selp.u32 q, " A ", q, t;\n" \
  "@start add.u32 %3, " S ", %" T17 ";\n" \
  ON_START(F) \
  "@start mov.u32 %5, 0;\n" \
  "@start mov.u32 %6, 0;\n" \
  "@start mov.f32 %7, 0f00000000;\n" \
  "not.pred t, start;\n" \
  "and.pred t, t, seeded;\n" \
  "or.pred seeded, t, seed;\n" \
  "mov.b32 nz, " N ";\n" \
  "@act mad.lo.u32 %5, q, 65536, %5;\n" \
  "@act add.u32 %5, %5, " A ";\n" \
  "@act mad.lo.u32 %6, " S ", q, %6;\n" \
  "@act add.rn.f32 %7, %7, nz;\n" \
  "@act add.u32 %4, " S ", 1;\n"
  #define CS_WALK(E2, ENTRY, M0, M1, LT, FEW, REC, HALF, SHIFT, T17, ON_FETCH, ON_EMIT, ON_START) \
  "{\n" \
  ".reg .pred hdr, ok, alive0, alive1, act, seed, start, emit, seeded, t;\n" \
  ".reg .u32 b0, b1, e, u, ad, lo, hi, gap, d, bal, i, x, m, q;\n" \
  ".reg .u32 s0, a0, c0, n0, f0, s1, a1, c1, n1, f1;\n" \
  ".reg .f32 nz;\n" \
  ".reg .u64 g;\n" \
  "setp.ne.u32 seeded, %8, 0;\n" \
  "setp.ne.u32 alive1, %" E2 ", 0;\n" \
  "mov.u32 a0, 0;\n" \
  "mov.u32 c0, 0;\n" \
  "mov.u32 n0, 0;\n" \
  "mov.u32 a1, 0;\n" \
  "mov.u32 c1, 0;\n" \
  "mov.u32 n1, 0;\n" \
  "mov.u32 b0, 0;\n" \
  "mov.u32 b1, 0;\n" \
  CS_FETCH("s0", "a0", "c0", "n0", "f0", "alive0", "alive1", E2, ENTRY, ON_FETCH) \
  "STEP:\n" \
  "vote.sync.ballot.b32 bal, alive0, 0xffffffff;\n" \
  "popc.b32 i, bal;\n" \
  "setp.le.u32 t, i, %" FEW ";\n" \
  "@t bra.uni DONE;\n" \
  CS_FETCH("s1", "a1", "c1", "n1", "f1", "alive1", "alive0", E2, ENTRY, ON_FETCH) \
  CS_USE("s0", "a0", "c0", "n0", "f0", "alive0", "NEXT0", M0, M1, LT, REC, HALF, SHIFT, T17, ON_EMIT, ON_START) \
  CS_FETCH("s0", "a0", "c0", "n0", "f0", "alive0", "alive1", E2, ENTRY, ON_FETCH) \
  CS_USE("s1", "a1", "c1", "n1", "f1", "alive1", "NEXT1", M0, M1, LT, REC, HALF, SHIFT, T17, ON_EMIT, ON_START) \
  "bra.uni STEP;\n" \
  "DONE:\n" \
  "@alive0 sub.u32 %0, %0, 1;\n" \
  "@alive0 sub.u32 %1, %1, 1;\n" \
  "selp.u32 %8, 1, 0, seeded;\n" \
  "selp.u32 %11, 1, 0, alive0;\n" \
  "}\n"
// The same with entries two steps ahead, for those in global memory: a step of the warps
// of a scheduler takes about 400 cycles, an entry from L2 more.  The two digis fetched
// last are used, not given back.
  #define CS_WALK_AHEAD(E2, ENTRY, M0, M1, LT, FEW, REC, HALF, SHIFT, T17, ON_FETCH, ON_EMIT, ON_START) \
  "{\n" \
  ".reg .pred hdr, ok, alive0, alive1, alive2, act, seed, start, emit, seeded, t;\n" \
  ".reg .u32 b0, b1, e, u, ad, lo, hi, gap, d, bal, i, x, m, q;\n" \
  ".reg .u32 s0, a0, c0, n0, f0, s1, a1, c1, n1, f1, s2, a2, c2, n2, f2;\n" \
  ".reg .f32 nz;\n" \
  ".reg .u64 g;\n" \
  "setp.ne.u32 seeded, %8, 0;\n" \
  "setp.ne.u32 alive2, %" E2 ", 0;\n" \
  "mov.u32 a0, 0;\n" \
  "mov.u32 c0, 0;\n" \
  "mov.u32 n0, 0;\n" \
  "mov.u32 a1, 0;\n" \
  "mov.u32 c1, 0;\n" \
  "mov.u32 n1, 0;\n" \
  "mov.u32 a2, 0;\n" \
  "mov.u32 c2, 0;\n" \
  "mov.u32 n2, 0;\n" \
  "mov.u32 b0, 0;\n" \
  "mov.u32 b1, 0;\n" \
  CS_FETCH("s0", "a0", "c0", "n0", "f0", "alive0", "alive2", E2, ENTRY, ON_FETCH) \
  CS_FETCH("s1", "a1", "c1", "n1", "f1", "alive1", "alive0", E2, ENTRY, ON_FETCH) \
  "STEP:\n" \
  "vote.sync.ballot.b32 bal, alive0, 0xffffffff;\n" \
  "popc.b32 i, bal;\n" \
  "setp.le.u32 t, i, %" FEW ";\n" \
  "@t bra.uni DONE;\n" \
  CS_FETCH("s2", "a2", "c2", "n2", "f2", "alive2", "alive1", E2, ENTRY, ON_FETCH) \
  CS_USE("s0", "a0", "c0", "n0", "f0", "alive0", "NEXT0", M0, M1, LT, REC, HALF, SHIFT, T17, ON_EMIT, ON_START) \
  CS_FETCH("s0", "a0", "c0", "n0", "f0", "alive0", "alive2", E2, ENTRY, ON_FETCH) \
  CS_USE("s1", "a1", "c1", "n1", "f1", "alive1", "NEXT1", M0, M1, LT, REC, HALF, SHIFT, T17, ON_EMIT, ON_START) \
  CS_FETCH("s1", "a1", "c1", "n1", "f1", "alive1", "alive0", E2, ENTRY, ON_FETCH) \
  CS_USE("s2", "a2", "c2", "n2", "f2", "alive2", "NEXT2", M0, M1, LT, REC, HALF, SHIFT, T17, ON_EMIT, ON_START) \
  "bra.uni STEP;\n" \
  "DONE:\n" \
  CS_USE("s0", "a0", "c0", "n0", "f0", "alive0", "NEXT3", M0, M1, LT, REC, HALF, SHIFT, T17, ON_EMIT, ON_START) \
  CS_USE("s1", "a1", "c1", "n1", "f1", "alive1", "NEXT4", M0, M1, LT, REC, HALF, SHIFT, T17, ON_EMIT, ON_START) \
  "selp.u32 %8, 1, 0, seeded;\n" \
  "selp.u32 %11, 1, 0, alive1;\n" \
  "}\n"
#define CS_NOTHING(F)
#define CS_FROM_FETCH(F) "mad.lo.u32 " F ", %2, 65536, %0;\n"
#define CS_FROM_START(F) "@start mov.u32 %12, " F ";\n"
#define CS_ENTRY13S(S, C, N, AL) "mad.lo.u32 ad, " S ", 8, %13;\n" "@" AL " ld.shared.v2.u32 {" C ", " N "}, [ad];\n"
#define CS_ENTRY13D(S, C, N, AL) "mad.wide.u32 g, " S ", 8, %13;\n" "@" AL " ld.global.nc.v2.u32 {" C ", " N "}, [g];\n"
#define CS_ENTRY14S(S, C, N, AL) "mad.lo.u32 ad, " S ", 8, %14;\n" "@" AL " ld.shared.v2.u32 {" C ", " N "}, [ad];\n"
#define CS_ENTRY14D(S, C, N, AL) "mad.wide.u32 g, " S ", 8, %14;\n" "@" AL " ld.global.nc.v2.u32 {" C ", " N "}, [g];\n"

template <bool AMP, bool DIRECT>
__device__ __forceinline__ bool walk_staged(Walk& k, uint32_t end2, const uint2* cal, int32_t m0, int32_t m1,
                                            uint32_t task17, uint32_t few, List& list) {
  const uint32_t lt = (1u << (threadIdx.x & 31)) - 1u;
  uint32_t walking;
  if (AMP && DIRECT) {
    asm volatile(CS_WALK_AHEAD("13", CS_ENTRY14D, "15", "16", "17", "18", "19", "20", "21", "22",
                         CS_FROM_FETCH,
                         "mad.wide.u32 g, i, 4, %23;\n"
                         "@emit st.global.u32 [g], %12;\n",
                         CS_FROM_START)
                 : "+r"(k.p), "+r"(k.strip), "+r"(k.strip_end), "+r"(k.first), "+r"(k.last1), "+r"(k.sums),
                   "+r"(k.moment), "+f"(k.n2), "+r"(k.seeded), "+r"(k.digis), "+r"(list.n), "=r"(walking),
                   "+r"(k.from)
                 : "r"(end2), "l"(cal), "r"(m0), "r"(m1), "r"(lt), "r"(few), "l"(list.rec),
                   "n"(1 << (kMulShift - 1)), "n"(kMulShift), "r"(task17), "l"(list.from)
                 : "memory");
  } else if (AMP) {
    asm volatile(CS_WALK("13", CS_ENTRY14S, "15", "16", "17", "18", "19", "20", "21", "22",
                         CS_FROM_FETCH,
                         "mad.wide.u32 g, i, 4, %23;\n"
                         "@emit st.global.u32 [g], %12;\n",
                         CS_FROM_START)
                 : "+r"(k.p), "+r"(k.strip), "+r"(k.strip_end), "+r"(k.first), "+r"(k.last1), "+r"(k.sums),
                   "+r"(k.moment), "+f"(k.n2), "+r"(k.seeded), "+r"(k.digis), "+r"(list.n), "=r"(walking),
                   "+r"(k.from)
                 : "r"(end2), "r"((uint32_t)__cvta_generic_to_shared(cal)), "r"(m0), "r"(m1), "r"(lt), "r"(few), "l"(list.rec),
                   "n"(1 << (kMulShift - 1)), "n"(kMulShift), "r"(task17), "l"(list.from)
                 : "memory");
  } else if (DIRECT) {
    asm volatile(CS_WALK_AHEAD("12", CS_ENTRY13D, "14", "15", "16", "17", "18", "19", "20", "21",
                         CS_NOTHING, "", CS_NOTHING)
                 : "+r"(k.p), "+r"(k.strip), "+r"(k.strip_end), "+r"(k.first), "+r"(k.last1), "+r"(k.sums),
                   "+r"(k.moment), "+f"(k.n2), "+r"(k.seeded), "+r"(k.digis), "+r"(list.n), "=r"(walking)
                 : "r"(end2), "l"(cal), "r"(m0), "r"(m1), "r"(lt), "r"(few), "l"(list.rec),
                   "n"(1 << (kMulShift - 1)), "n"(kMulShift), "r"(task17)
                 : "memory");
  } else {
    asm volatile(CS_WALK("12", CS_ENTRY13S, "14", "15", "16", "17", "18", "19", "20", "21",
                         CS_NOTHING, "", CS_NOTHING)
                 : "+r"(k.p), "+r"(k.strip), "+r"(k.strip_end), "+r"(k.first), "+r"(k.last1), "+r"(k.sums),
                   "+r"(k.moment), "+f"(k.n2), "+r"(k.seeded), "+r"(k.digis), "+r"(list.n), "=r"(walking)
                 : "r"(end2), "r"((uint32_t)__cvta_generic_to_shared(cal)), "r"(m0), "r"(m1), "r"(lt), "r"(few), "l"(list.rec),
                   "n"(1 << (kMulShift - 1)), "n"(kMulShift), "r"(task17)
                 : "memory");
  }
  return walking != 0;
}
#undef CS_WALK
#undef CS_WALK_AHEAD
#undef CS_FETCH
#undef CS_USE
#undef CS_NOTHING
#undef CS_FROM_FETCH
#undef CS_FROM_START
#undef CS_ENTRY13S
#undef CS_ENTRY13D
#undef CS_ENTRY14S
#undef CS_ENTRY14D

// The same walk for any record: read in place from anywhere (a unit larger than the
// staging buffer), APVs without a multiplier dividing.  One channel per lane to the
// record's end (`end` == p: none).
template <bool AMP>
__device__ void walk_any(Walk& k, const uint8_t* src, uint32_t end, const uint2* cal, int32_t m0, int32_t m1,
                         uint32_t task17, List& list) {
  for (;;) {
    const bool hdr = k.strip == k.strip_end;
    uint32_t b0 = 0, b1 = 0;
    if (hdr && k.p + 2 <= end) {
      b0 = src[k.p];
      b1 = src[k.p + 1];
    }
    const bool ok = hdr && k.p + 2 + b1 <= end && b0 + b1 <= (uint32_t)kStrips && b1 != 0 && b0 >= k.strip;
    const bool alive = !hdr || ok;
    if (!__any_sync(0xffffffffu, alive)) break;
    if (ok) {
      k.strip = b0;
      k.strip_end = b0 + b1;
      k.p += 2;
    }
    const uint32_t s = k.strip;
    uint32_t a = 0;
    uint2 c = make_uint2(0u, 0u);
    if (alive) {
      a = src[k.p++];
      c = cal[s];
      k.strip++;
      k.digis++;
    }
    const bool act = a > (c.x & 255u), seed = a > ((c.x >> 8) & 255u);  // a lane that has stopped: 0, never active
    const bool start = act && s - k.last1 >= (c.x >> 16);
    list.append<AMP>(start && k.seeded, k.record(), k.from);
    if (act) {
      const uint32_t q = charge(a, s < (uint32_t)kApv ? m0 : m1);
      if (start) {
        k.first = s + task17;
        k.from = (k.strip_end << 16) + k.p;
        k.sums = k.moment = k.seeded = 0;
        k.n2 = 0.f;
      }
      k.sums += (q << 16) + a;
      k.moment += s * q;
      k.n2 = __fadd_rn(k.n2, __uint_as_float(c.y));
      k.seeded |= seed ? 1u : 0u;
      k.last1 = s + 1u;
    }
  }
}

// What a lane that stopped at byte p of its record, before its end, found there:
// the first rule that the header at p breaks.  rd reads a byte.
template <typename Rd>
__device__ __forceinline__ uint32_t stop_status(const Walk& k, uint32_t end, Rd rd) {
  if (k.p + 2 > end) return SST_CH_TRUNC;
  const uint32_t f = rd(k.p), wd = rd(k.p + 1);
  return wd - 1u > (uint32_t)kStrips - 1u - f ? (uint32_t)SST_CH_RUN_RANGE
         : f < k.strip                        ? (uint32_t)SST_CH_RUN_ORDER
                                              : (uint32_t)SST_CH_TRUNC;
}

// A record's strips [lo, hi], widened over up to max_adj adjacent bad strips of module
// det at either end.
__device__ __forceinline__ void record_strips(uint4 r, const KParams& kp, uint32_t det, int* lo, int* hi) {
  *lo = (int)(r.x & 255u);
  *hi = (int)((r.x >> 8) & 511u) - 1;
  if (kp.max_adj > 0) {
    const uint32_t* m = kp.badmask + (size_t)det * kMaskWords;
    for (int k = 0; k < kp.max_adj && *lo > 0 && bit(m, *lo - 1); k++) --*lo;
    for (int k = 0; k < kp.max_adj && *hi + 1 < kStrips && bit(m, *hi + 1); k++) ++*hi;
  }
}

// Amplitude staging of a launch (rec null: no amplitudes).
struct Amps {
  uint32_t* spill = nullptr;      // per warp of the grid, kAmpSpill words (List::from)
  uint8_t* bytes = nullptr;       // staged amplitudes, sliced per event like the output
  uint32_t* first = nullptr;      // per staged cluster: its first amplitude within its segment
  const uint64_t* off = nullptr;  // [n_events + 1] event slices
  uint64_t cap = 0;               // bytes of staging and of output
  uint32_t* alloc = nullptr;      // allocation counter per event
  uint32_t* seg_cnt = nullptr;    // per segment: amplitudes stored (0 when they did not fit)
  uint32_t* seg_start = nullptr;  // per segment: offset in the event's slice, or kNoAmp
};
// Event e's slice [a, b) of the amplitude arrays.
__device__ __forceinline__ void amp_slice(const uint64_t* off, uint64_t cap, uint32_t e, uint32_t* a, uint32_t* b) {
  uint64_t lo = off[e], hi = off[e + 1] < cap ? off[e + 1] : cap;  // cap is below 2^32
  if (lo > hi) lo = hi;
  *a = (uint32_t)lo;
  *b = (uint32_t)hi;
}

// The channels of a warp's tasks.  Tile: every slot has the same C channels (of many
// events), in shared memory.  DIRECT: the slots are FE units of one FED, one after the
// other, in global memory; SPAN: their bytes are copied as one piece.
template <int C, bool DIRECT, bool SPAN = false>
struct Channels {
  static constexpr bool kDirect = DIRECT, kSpan = SPAN;
  const uint2* cal;  // calibration entries of the first channel
  const int2* mul;   // APV multipliers, two per channel
  uint32_t ch0;      // module id of the first channel
  // channel of task t, slots counted from slot `done`
  __device__ __forceinline__ uint32_t of(uint32_t t, int done) const {
    return DIRECT ? (uint32_t)done * C + t : t % C;
  }
};

// Cluster threshold of every record and the kept ones' places within their
// channel: record i's z becomes the number of kept records of its channel before
// it, or kNotKept; w.kept counts them.  A channel's records are in strip order.
// AMP: the strips of those before are added to z at bit 8, and w.task (free by now) sums
// each channel's.
template <bool AMP, class W, class Chans>
__device__ __forceinline__ void rank_records(W& w, const List& list, const KParams& kp, const Chans& chans, int done) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  for (int i = lane; i < W::kTasks / 4; i += 32) reinterpret_cast<uint32_t*>(w.kept)[i] = 0;
  if (AMP)
    for (int i = lane; i < W::kTasks; i += 32) w.task[i] = 0;
  __syncwarp();
  const Threshold thr(kp.t_cluster);
  const uint4 none = make_uint4(0u, 0u, 0x7f800000u, 0u);
  uint4 ahead = (uint32_t)lane < list.n ? list.rec[lane] : none;
  for (uint32_t i = lane; i - lane < list.n; i += 32) {
    const uint4 r = ahead;
    if (i - lane + 32 < list.n) ahead = i + 32 < list.n ? list.rec[i + 32] : none;
    const bool pass = thr.pass(r.y & 0xFFFFu, __uint_as_float(r.z));
    const uint32_t t = r.x >> 17;
    const unsigned same = __match_any_sync(0xffffffffu, pass ? t : 128u);
    uint32_t rank = (pass ? (uint32_t)w.kept[t] : 0u) + __popc(same & lt), z = rank;
    if (AMP) {
      int lo = 0, hi = -1;
      if (pass) record_strips(r, kp, chans.ch0 + chans.of(t, done), &lo, &hi);
      const uint32_t wd = (uint32_t)(hi - lo + 1);
      uint32_t before = pass ? w.task[t] : 0u;
      for (unsigned m = pass ? same & lt : 0u; __any_sync(0xffffffffu, m != 0); m &= m - 1u) {
        const uint32_t v = __shfl_sync(0xffffffffu, wd, m ? __ffs(m) - 1 : 0);
        if (m) before += v;
      }
      z |= before << 8;
      __syncwarp();
      if (pass && (same >> lane) == 1u) w.task[t] = before + wd;
    } else {
      __syncwarp();
    }
    if (pass && (same >> lane) == 1u) w.kept[t] = (uint8_t)(rank + 1u);  // the channel's last record here
    if (i < list.n) list.rec[i].z = pass ? z : kNotKept;
    __syncwarp();
  }
}

// Staged cluster: 8 bytes, the centroid's division left to the ordering pass.
// x = lowest strip | width - 1 << 8 | charge << 16; y = moment about the lowest
// strip (24 bits: at most 255 x 65,280) | channel in the segment << 24.
__device__ __forceinline__ uint2 staged_cluster(uint32_t lo, uint32_t wd, uint32_t q, uint32_t moment, uint32_t c) {
  return make_uint2(lo | ((wd - 1u) << 8) | (q << 16), moment | (c << 24));
}

// Writes the kept clusters to the events' staging slices (w.task: place of each
// channel's first).  det(t) is the module of channel t.
template <int C, class W, typename Det>
__device__ __forceinline__ void write_records(const W& w, const List& list, const KParams& kp, uint2* stage, Det det) {
  const int lane = threadIdx.x & 31;
  uint4 ahead = make_uint4(0u, 0u, 0u, 0u);
  if ((uint32_t)lane < list.n) ahead = list.rec[lane];
  for (uint32_t i = lane; i < list.n; i += 32) {
    const uint4 r = ahead;
    if (i + 32 < list.n) ahead = list.rec[i + 32];
    if (r.z == kNotKept) continue;
    const uint32_t t = r.x >> 17, slot = t / C;
    const uint32_t pos = w.task[t] + r.z;
    if (pos >= w.slot.room[slot]) continue;
    int lo, hi;
    record_strips(r, kp, det(t), &lo, &hi);
    const uint32_t q = r.y >> 16;
    stage[w.base[slot] + pos] =
        staged_cluster((uint32_t)lo, (uint32_t)(hi - lo + 1), q, r.w - (uint32_t)lo * q, t - slot * C);
  }
}

// write_records for clusters with amplitudes.  `rel` (per task): the strips of the slot's
// channels before it; w.slot.nbad: where the slot's amplitudes are staged, or kNoAmp.  A
// cluster's amplitudes: 0 for every strip but its active digis, whose charges are formed
// again from the record's bytes (rd; `shift` makes an index of a Walk::from byte) and
// the calibration entries.
template <int C, class W, class Chans, typename Rd>
__device__ __forceinline__ void write_amplitudes(const W& w, const List& list, const KParams& kp, uint2* stage,
                                                 const Amps& am, const uint32_t* rel, const Chans& chans, int done,
                                                 uint32_t shift, Rd rd) {
  const int lane = threadIdx.x & 31;
  uint4 ahead = make_uint4(0u, 0u, kNotKept, 0u);
  uint32_t from_ahead = 0;
  if ((uint32_t)lane < list.n) {
    ahead = list.rec[lane];
    from_ahead = list.from[lane];
  }
  for (uint32_t i = lane; i < list.n; i += 32) {
    const uint4 r = ahead;
    const uint32_t from = from_ahead;
    if (i + 32 < list.n) {
      ahead = list.rec[i + 32];
      from_ahead = list.from[i + 32];
    }
    if (r.z == kNotKept) continue;
    const uint32_t t = r.x >> 17, slot = t / C, c = chans.of(t, done);
    const uint32_t pos = w.task[t] + (r.z & 255u), first = rel[t] + (r.z >> 8);
    int lo, hi;
    record_strips(r, kp, chans.ch0 + c, &lo, &hi);
    const uint32_t q = r.y >> 16;
    if (pos < w.slot.room[slot]) {
      stage[w.base[slot] + pos] =
          staged_cluster((uint32_t)lo, (uint32_t)(hi - lo + 1), q, r.w - (uint32_t)lo * q, t - slot * C);
      am.first[w.base[slot] + pos] = first;
    }
    if (w.slot.nbad[slot] == kNoAmp) continue;
    uint8_t* d = am.bytes + (size_t)w.slot.nbad[slot] + first;
    uint32_t p = ((from + shift) & 0xFFFFu) - 1u, run_end = from >> 16, next = r.x & 255u;  // next: strip of the digi at p
    const uint32_t last1 = (r.x >> 8) & 511u;
    const uint2* cal = chans.cal + c * kStrips;
    const int2 mul = chans.mul[c];
    for (uint32_t st = (uint32_t)lo; st <= (uint32_t)hi; st++) {
      uint32_t v = 0;
      if (st == next && st < last1) {
        const uint32_t a = rd(p++);
        if (a > (cal[st].x & 255u)) v = charge(a, st < (uint32_t)kApv ? mul.x : mul.y);
        if (++next == run_end && next < last1) {
          next = rd(p);
          run_end = next + rd(p + 1);
          p += 2;
        }
      }
      *d++ = (uint8_t)v;
    }
  }
}

// The order in which the channels are walked, longest record first: the lanes of a
// warp then finish at about the same time.  A counting sort by length / 4 (all
// records of 124 bytes and more in one bin).
template <class W>
__device__ __forceinline__ void order_tasks(W& w, int n_task) {
  constexpr int kJ = (W::kTasks + 31) / 32;
  const int lane = threadIdx.x & 31;
  uint32_t* bins = w.bins;
  bins[lane] = 0;
  __syncwarp();
  uint32_t bin[kJ], rank[kJ];
#pragma unroll
  for (int j = 0; j < kJ; j++) {
    const int t = lane + 32 * j;
    if (t < n_task) {
      const uint32_t l = w.task[t] >> 18;
      bin[j] = l < 31u ? 31u - l : 0u;
      rank[j] = atomicAdd(&bins[bin[j]], 1u);
    }
  }
  __syncwarp();
  const uint32_t v = bins[lane];
  uint32_t x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  bins[lane] = x - v;
  __syncwarp();
#pragma unroll
  for (int j = 0; j < kJ; j++) {
    const int t = lane + 32 * j;
    if (t < n_task) w.order[bins[bin[j]] + rank[j]] = (uint8_t)t;
  }
  __syncwarp();
}

// Where a slot's FE unit is (one lane per slot).
struct SlotSrc {
  const uint8_t* src;  // first byte of the unit's records
  uint32_t len;        // their bytes (0: no data)
  uint32_t status;     // SST_CH_FED_HDR when the FED record is corrupt or out of range
  bool data;           // the FED record is there and its header is valid
};

// The channel length chain of one FE unit of len bytes from p (the paper's map of
// channel locations): each length at least 3, within the unit, and all of them adding
// up to the unit's length; otherwise false, and no channel of the unit is read.
// put(k, pos, length) takes channel k (it may have been called when the chain breaks).
template <typename Rd, typename Put>
__device__ __forceinline__ bool walk_lengths(uint32_t p, uint32_t len, Rd rd, Put put) {
  const uint32_t end = p + len;
  bool good = true;
#pragma unroll
  for (int k = 0; k < kChPerFe; k++) {
    good = good && p + 2 <= end;
    uint32_t l = 0;
    if (good) l = rd(p) | (rd(p + 1) << 8);
    good = good && l >= 3 && p + l <= end;
    if (good) {
      put(k, p, l);
      p += l;
    }
  }
  return good && p == end;
}

// Unpacks and clusters n <= 32 slots (lane s < n holds slot s's FE unit in `me`, its event
// in `e`, its segment index in `seg`): channels c0 .. c0 + C - 1 of each unit.
// any_div: an APV of theirs has no multiplier.  before_rank() runs between the walk and
// the rest.
template <bool AMP, int C, class W, class Chans, typename Hook>
__device__ void process_slots(W& w, int n, int c0, const SlotSrc& me, uint32_t e, size_t seg, const KParams& kp,
                              const uint64_t* __restrict__ clu_off, uint64_t out_cap, sst_event_status* status,
                              uint2* stage, uint32_t* ev_alloc, uint32_t* seg_cnt, uint32_t* seg_start, uint4* spill,
                              const Chans& chans, bool any_div, const Amps& am,
                              uint32_t* amp_spill, Hook before_rank) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  constexpr int kL = C / 3;  // lanes per slot when a lane sums three channels
  uint64_t off = 0, end = 0;
  if (lane < n) {
    off = clu_off[e];
    end = clu_off[e + 1] < out_cap ? clu_off[e + 1] : out_cap;
  }
  const uint32_t padded = (me.len + 7u) & ~7u;
  int done = 0;
  while (done < n) {
    // the next slots whose bytes fit the staging buffer together; a unit larger
    // than the buffer is taken alone and read in place
    uint32_t x = lane >= done && lane < n ? padded : 0u;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    const unsigned fit = __ballot_sync(0xffffffffu, lane >= done && lane < n && x <= (uint32_t)W::kBuf);
    int m = __popc(fit);
    m = m < W::kSlots ? m : W::kSlots;
    if (m < n - done && m > (n - done + 1) / 2) m = (n - done + 1) / 2;  // two halves rather than most and a rest
    const bool staged = m > 0;
    if (!staged) m = 1;
    const bool mine = lane >= done && lane < done + m;
    const uint32_t at = x - padded;  // my unit's place in the buffer
    const uint8_t* src0 = reinterpret_cast<const uint8_t*>(
        __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(me.src), done));
    if (staged && Chans::kSpan) {
      // one copy of the units by the whole warp.  (From pinned host memory in pieces of 688
      // bytes 188 GB/s, against 175 by half warps, unit by unit; from device memory it is
      // within 3% either way, and 10% slower with amplitudes.)
      const uint32_t len = __shfl_sync(0xffffffffu, x, done + m - 1);
      if ((reinterpret_cast<uintptr_t>(src0) & 7u) == 0) {
        for (uint32_t i = lane; i < len >> 3; i += 32)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                           (uint32_t)__cvta_generic_to_shared(w.buf + 8 * i)),
                       "l"(src0 + 8 * i)
                       : "memory");
      } else {
        for (uint32_t i = lane; i < len; i += 32) w.buf[i] = __ldg(src0 + i);
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (staged) {
      // two units at a time, half a warp each (128 bytes a request)
      for (int k = 0; k < m; k += 2) {
        const int s = done + k + (lane >> 4);
        const int from = s < done + m ? s : done;
        const uint8_t* g = reinterpret_cast<const uint8_t*>(
            __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(me.src), from));
        const uint32_t len_s = __shfl_sync(0xffffffffu, me.len, from);
        const uint32_t len = s < done + m ? len_s : 0u;
        uint8_t* dst = w.buf + __shfl_sync(0xffffffffu, at, from);
        if ((reinterpret_cast<uintptr_t>(g) & 7u) == 0) {
          const uint32_t nv = (len + 7u) >> 3;  // whole 8-byte words; padding bytes exist up to the next 8
          for (uint32_t i = lane & 15; i < nv; i += 16)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                             (uint32_t)__cvta_generic_to_shared(dst + 8 * i)),
                         "l"(g + 8 * i)
                         : "memory");
        } else {
          for (uint32_t i = lane & 15; i < len; i += 16) dst[i] = __ldg(g + i);
        }
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
    }
    __syncwarp();
    uint32_t st = 0;
    if (mine) {
      const int s = lane - done;
      bool good = false;
      auto put = [&](int k, uint32_t pos, uint32_t l) {
        if (k >= c0 && k < c0 + C) w.task[s * C + k - c0] = pos | (l << 16);
      };
      if (me.data) {
        if (staged)
          good = walk_lengths(at, me.len, [&](uint32_t i) { return (uint32_t)w.buf[i]; }, put);
        else
          good = walk_lengths(0u, me.len, [&](uint32_t i) { return (uint32_t)src0[i]; }, put);
      }
      if (!good)
        for (int k = 0; k < C; k++) w.task[s * C + k] = 0u;
      st = good ? 0u : me.data ? (uint32_t)SST_CH_FRAMING : me.status;
      w.base[s] = off < out_cap ? off : 0;
    }
    __syncwarp();
    const int n_task = m * C;
    order_tasks(w, n_task);
    const uint32_t room = end > off ? (uint32_t)(end - off < 0xFFFFFFFFull ? end - off : 0xFFFFFFFFull) : 0u;
    if (mine) {
      w.slot.room[lane - done] = room;
      w.slot.digis[lane - done] = 0;
      w.slot.flags[lane - done] = st;
      w.slot.nbad[lane - done] = st ? (uint32_t)C : 0u;
    }
    __syncwarp();
    List list{spill, amp_spill, 0u};
    // A channel found corrupt (its lane calls with err): its status, and its records,
    // among those from `from` on, are dropped.
    auto corrupt = [&](uint32_t t, uint32_t err) {
      __syncwarp();
      if (err) {
        atomicOr(&w.slot.flags[t / C], err);
        atomicAdd(&w.slot.nbad[t / C], 1u);
        for (uint32_t i = 0; i < list.n; i++)
          if ((list.rec[i].x >> 17) == t) list.rec[i].z = 0x7f800000u;  // noise^2 infinite: below every threshold
      }
      __syncwarp();
    };
    // The same at src, byte by byte, for any record and any APV.
    auto walk_in_place = [&](int t0, int t1, const uint8_t* src) {
      for (int r0 = t0; r0 < t1; r0 += 32) {
        uint32_t t = 0, tk = 0;
        if (r0 + lane < t1) {
          t = w.order[r0 + lane];
          tk = w.task[t];
        }
        const uint32_t pos = tk & 0xFFFFu, len = tk >> 16;
        const bool has = len >= 3u, code = has && src[pos + 2] == SST_ZS_CODE;
        const uint32_t c = chans.of(t, done);
        const int2 mm = chans.mul[c];
        Walk k;
        k.begin(pos + 3u);
        const uint32_t rec_end = code ? pos + len : 0u;
        walk_any<AMP>(k, src, rec_end, chans.cal + c * kStrips, mm.x, mm.y, t << 17, list);
        const uint32_t err = !has ? 0u
                             : !code ? (uint32_t)SST_CH_BAD_CODE
                             : k.p != rec_end ? stop_status(k, rec_end, [&](uint32_t i) { return (uint32_t)src[i]; })
                                              : 0u;
        list.append<AMP>(has && !err && k.seeded, k.record(), k.from);
        if (has && !err) atomicAdd(&w.slot.digis[t / C], k.digis);
        if (__any_sync(0xffffffffu, err != 0u)) corrupt(t, err);
      }
    };
    const uint32_t buf0 = (uint32_t)__cvta_generic_to_shared(w.buf);
    // Walks channels order[t0] .. order[t1 - 1], whose records are in the buffer `shift`
    // bytes before their positions.
    auto walk_fast = [&](int t0, int t1, uint32_t shift) {
      int next = t0;                      // channels taken
      bool walking = false, has = false;  // the lane has a channel record: task t, bytes up to rec_end
      uint32_t t = 0, rec_end = 0;
      const uint2* cal = chans.cal;
      int2 mm = make_int2(0, 0);
      Walk k;
      k.begin(buf0);
      for (;;) {
        // lanes at their record's end: its last candidate, its digis
        const bool ended = has && !walking;
        const bool bad = ended && k.p != rec_end;
        if (ended && !bad) atomicAdd(&w.slot.digis[t / C], k.digis);
        list.append<AMP>(ended && !bad && k.seeded, k.record(), k.from);
        if (__any_sync(0xffffffffu, bad))
          corrupt(t, !bad ? 0u
                     : rec_end == 0u
                         ? (uint32_t)SST_CH_BAD_CODE
                         : stop_status(k, rec_end, [&](uint32_t i) { return (uint32_t)w.buf[i - buf0]; }));
        // the next channels
        const unsigned idle = __ballot_sync(0xffffffffu, !walking);
        if (!walking) {
          const int i = next + __popc(idle & lt);
          has = i < t1;
          uint32_t tk = shift;
          if (has) {
            t = w.order[i];
            tk = w.task[t];
          }
          const uint32_t pos = (tk & 0xFFFFu) - shift, len = tk >> 16, c = chans.of(t, done);
          has = len >= 3u;
          cal = chans.cal + c * kStrips;
          mm = chans.mul[c];
          k.begin(buf0 + pos + 3u);
          rec_end = has && w.buf[pos + 2u] == SST_ZS_CODE ? buf0 + pos + len : 0u;  // 0: stops at once
        }
        next += __popc(idle);
        if (!__any_sync(0xffffffffu, has)) break;
        walking = walk_staged<AMP, Chans::kDirect>(k, rec_end ? rec_end - 2u : 0u, cal, mm.x, mm.y, t << 17,
                              next < t1 ? (uint32_t)kRefill : 0u, list);
      }
    };
    if (staged && !any_div) {
      walk_fast(0, n_task, 0);
    } else if (!any_div) {
      // one FE unit larger than the buffer: as many of its channels at a time as fit
      if (lane < C) w.order[lane] = (uint8_t)lane;
      __syncwarp();
      for (int c = 0; c < C;) {
        const uint32_t p0 = (w.task[c] & 0xFFFFu) & ~7u;
        uint32_t end = p0;
        int c1 = c;
        while (c1 < C && (w.task[c1] & 0xFFFFu) + (w.task[c1] >> 16) - p0 <= (uint32_t)W::kBuf) {
          end = max(end, (w.task[c1] & 0xFFFFu) + (w.task[c1] >> 16));
          c1++;
        }
        if (c1 == c) {  // a record longer than the buffer (no valid one is)
          walk_in_place(c, c + 1, src0);
          c1 = c + 1;
        } else {
          const uint8_t* g = src0 + p0;
          if ((reinterpret_cast<uintptr_t>(g) & 7u) == 0) {
            for (uint32_t i = lane; i < (end - p0 + 7u) / 8u; i += 32)
              asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(buf0 + 8 * i), "l"(g + 8 * i) : "memory");
          } else {
            for (uint32_t i = lane; i < end - p0; i += 32) w.buf[i] = __ldg(g + i);
          }
          asm volatile("cp.async.wait_all;" ::: "memory");
          __syncwarp();
          const uint32_t n0 = list.n;
          walk_fast(c, c1, p0);
          __syncwarp();
          if (AMP)  // bytes of the unit, not of the buffer
            for (uint32_t i = n0 + lane; i < list.n; i += 32)
              list.from[i] = (list.from[i] & 0xFFFF0000u) | ((list.from[i] - buf0 + p0) & 0xFFFFu);
          __syncwarp();
        }
        c = c1;
      }
    } else {
      walk_in_place(0, n_task, staged ? w.buf : src0);
    }
    __syncwarp();
    if (done + m >= n) before_rank();
    rank_records<AMP>(w, list, kp, chans, done);
    // places: each lane sums three channels, kL lanes make a slot
    const bool sums3 = 3 * lane < W::kTasks;
    const uint32_t k0 = sums3 ? w.kept[3 * lane] : 0u, k1 = sums3 ? w.kept[3 * lane + 1] : 0u;
    const uint32_t sum = k0 + k1 + (sums3 ? w.kept[3 * lane + 2] : 0u);
    uint32_t incl = sum;
#pragma unroll
    for (int d = 1; d < kL; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d, kL);
      if ((lane & (kL - 1)) >= d) incl += y;
    }
    const uint32_t found = __shfl_sync(0xffffffffu, incl, (kL * (lane - done) + kL - 1) & 31);  // of my slot
    // the strips of their kept clusters, the same way
    uint32_t a0 = 0, a1 = 0, asum = 0, aincl = 0, strips = 0;
    if (AMP) {
      if (sums3) {
        a0 = w.task[3 * lane];
        a1 = w.task[3 * lane + 1];
        asum = a0 + a1 + w.task[3 * lane + 2];
      }
      aincl = asum;
#pragma unroll
      for (int d = 1; d < kL; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, aincl, d, kL);
        if ((lane & (kL - 1)) >= d) aincl += y;
      }
      strips = __shfl_sync(0xffffffffu, aincl, (kL * (lane - done) + kL - 1) & 31);
    }
    uint32_t start = 0;
    if (mine) {
      const uint32_t astart = AMP && strips ? atomicAdd(am.alloc + counter_at(e), strips) : 0u;
      start = found ? atomicAdd(ev_alloc + counter_at(e), found) : 0u;
      const uint32_t fits = start < room ? (found < room - start ? found : room - start) : 0u;
      uint32_t fl = w.slot.flags[lane - done];
      if (fits < found) fl |= SST_EV_CLUSTER_CAPACITY;
      const uint32_t nb = w.slot.nbad[lane - done], nd = w.slot.digis[lane - done];
      if (AMP) {
        uint32_t lo, hi;
        amp_slice(am.off, am.cap, e, &lo, &hi);
        const bool ok = (uint64_t)astart + strips <= hi - lo;
        if (!ok) fl |= SST_EV_AMP_CAPACITY;
        am.seg_cnt[seg] = ok ? strips : 0u;
        am.seg_start[seg] = ok ? astart : kNoAmp;
        w.slot.nbad[lane - done] = ok ? lo + astart : kNoAmp;
      }
      if (fl) atomicOr(&status[e].flags, fl);
      if (nb) atomicAdd(&status[e].n_bad_channels, nb);
      if (nd) atomicAdd(&status[e].n_digi, nd);
      seg_cnt[seg] = fits;
      seg_start[seg] = start;
    }
    const uint32_t place = __shfl_sync(0xffffffffu, start, (done + lane / kL) & 31) + incl - sum;
    uint32_t* rel = list.from + kSpillRecords;
    if (sums3) {
      w.task[3 * lane] = place;
      w.task[3 * lane + 1] = place + k0;
      w.task[3 * lane + 2] = place + k0 + k1;
      if (AMP) {
        rel[3 * lane] = aincl - asum;
        rel[3 * lane + 1] = aincl - asum + a0;
        rel[3 * lane + 2] = aincl - asum + a0 + a1;
      }
    }
    __syncwarp();
    if (AMP) {
      // (the fast walk's bytes are counted by shared address, of which 16 bits are enough)
      write_amplitudes<C>(w, list, kp, stage, am, rel, chans, done,
                          staged && !any_div ? 0u - (uint32_t)__cvta_generic_to_shared(w.buf) : 0u,
                          [&](uint32_t i) { return staged ? (uint32_t)w.buf[i] : (uint32_t)src0[i]; });
    } else {
      write_records<C>(w, list, kp, stage, [&](uint32_t tt) { return chans.ch0 + chans.of(tt, done); });
    }
    __syncwarp();
    done += m;
  }
}

}  // namespace cs

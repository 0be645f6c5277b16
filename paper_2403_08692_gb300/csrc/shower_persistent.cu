// Persistent shower form: one launch runs every event to the cutoff.
//
// Each warp keeps a pool of kSlots events whose state (ln t, hash, cycle, the
// screen's dipoles) stays in shared memory.  A veto cycle takes up to 32
// runnable events, one per lane:
//  1. Screen.  The trials of the warp's events are generated 32 splitters at
//     a time, whichever events they belong to (screen_warp), so events of
//     different sizes share a warp with no lane waiting for the largest, and
//     the last events of a launch spread over all lanes.
//  2. Decide.  Each lane settles its event's winner (FP64 scale), cutoff and
//     veto.  An event with an accepted emission waits; a finished one leaves.
// Once enough emissions wait, the block's warps generate them together,
// packed into as few warps as hold them (four lanes each where that is
// fewer than a warp a scheduler), and refresh the dipoles they moved with all
// threads.  Slots of events that left are written back and refilled
// from a global event cursor.  Events therefore leave as soon as they finish
// -- the paper's cutoff inefficiency (Sec. 2, Fig. 3: finished events wait
// for the last one) disappears.
//
// What bounds it, and why this shape.  FP64 instructions hold the SM's FP64
// pipe for 16 cycles whatever their active lanes, so the emissions (about 300
// of them each with their dipoles, against 14 per cycle) have to fill their
// warps: 32 of a warp's 64 events can wait while the others run, and the
// block packs them (19 -> 27 of 32 lanes on FP64 instructions).  The kernel's
// code is some 50 KB in its hot parts, more than the instruction cache next to
// the SM: warps that wandered through it each on their own stalled for
// instructions 7 of every 16 cycles; a block's warps meet before every
// emission turn and vote, so they run the same part at the same time (0.3 of
// 11).  Keeping the state in shared memory leaves one 32-byte record per
// cycle and event to global memory.  Measured (GB300, shower kernel alone;
// before: block pools of one or two events per thread, each event's trials
// in one thread, state in global memory): 10^6 LEP events 7.39 -> 5.33 ms,
// 10^5 1.31 -> 0.88 ms, 10^5 at 200 GeV and t_C = 0.5 3.30 -> 2.3 ms, 100
// events 0.54 -> 0.19 ms.  At 3x10^5 events the FP64 pipe is busy 43 % of the
// time and 37 % of the issue slots are used; 20 or 24 resident warps (fewer
// registers) and pools of 40 to 56 events were no faster.
//
// Nothing waits on another block: a block ends when its pools are empty and
// the cursor has passed the last event.  Every event stops after at most
// max_steps cycles (step-limit status), so the launch always terminates.
// The draws are keyed by (seed, event, cycle) and the winner, cutoff and veto
// are the plain form's code, so both forms give identical events.
#include <algorithm>

#include "gaps_launch.hpp"
#include "shower_cycle.cuh"

namespace gaps {

namespace {

// Events of a warp's pool: 32 can run while 32 wait for their emission, so
// both the cycles and the emissions fill the warp.
constexpr int kSlots = 64;
// The register budget is set for 16 warps per SM.
constexpr int kMaxThreads = 512;
// Warp schedulers of an SM.
constexpr int kSchedulers = 4;
// Veto cycles a warp runs between two votes of its block (1 to 8 were alike).
constexpr int kTurns = 3;

// Dipoles with phase space kept per event in shared memory; an event with
// more takes its screen's inputs from the record.  Six hold nearly every LEP
// event; 8 or 4 were 5 and 14 % slower for the persistent form at 10^6 LEP
// events (less first-level cache, more events in the record).  Event-cycles in
// the record: LEP 0.8 %, 200 GeV 1.8 % at t_C = 2 GeV^2 and 8.5 % at 0.5, 500
// GeV 12 % at 1 and 19 % at 0.5; other counts were not timed there.
constexpr int kDips = 6;
constexpr uint8_t kInRecord = 255;

// What the screens of a warp read of its events.
struct ScreenPool {
  float dip_x[kDips][kSlots], dip_y[kDips][kSlots];  // the dipoles' screen entries
  uint32_t dip_m[kDips][kSlots];                     // slot on side 0 | slot on side 1 << 8 | gluons << 16, 17
  int32_t ev[kSlots];
  // the event's splitters, dipole * 2 + side: those with a gluon's kernels
  // from the front, those with one trial from the back; how many of either
  // kind (n_all = kInRecord: in the record)
  uint8_t split[2 * kDips][kSlots];
  uint8_t n_all[kSlots], n_one[kSlots], n[kSlots];
  uint8_t owner[64];
};
// The screens' results, per lane.
struct ScreenResults {
  uint32_t best[32], second[32], code[32], hi[32], lo[32];
  float invc[32];
};
__device__ __forceinline__ unsigned lanes_below(int lane) { return (1u << lane) - 1u; }

// Lanes of a warp per event for up to 32 events: a power of two.
__device__ __forceinline__ int lanes_each(int events) { return 1 << min(max(__clz(events - 1) - 27, 0), 5); }

// Splitters (sides of dipoles with phase space) of an event, and those of
// them that are gluons.
struct SideCounts {
  int all, gluons;
};

// Load the screen's dipoles of the events in slots q of the warp's first 32 /
// L lanes (q < 0: none), L lanes per event: those with phase space, each once
// (from its colour end).  Returns each such lane its event's counts.  The
// partons' data are loaded side by side over the lanes, so a few events take
// one or two memory latencies whatever their size.  Every lane of the warp
// must call it.
template <int kMode>
__device__ __forceinline__ SideCounts load_dipoles(const DevParams& P0, const Events& E, ScreenPool& w, int q, int job,
                                                   int L) {
  const int lane = static_cast<int>(threadIdx.x & 31);
  const int el = lane / L, sub = lane - el * L;
  const unsigned group = (L == 32 ? 0xffffffffu : (1u << L) - 1u) << (el * L);
  const unsigned before = group & lanes_below(lane);
  const int eq = __shfl_sync(0xffffffffu, q, el);
  const bool combined = per_dipole<kMode>(job_params<kJobPhysics<kMode>>(P0, E, __shfl_sync(0xffffffffu, job, el)));
  const int64_t ev = eq >= 0 ? w.ev[eq] : 0;
  const int n = eq >= 0 ? w.n[eq] : 0;
  const int rounds = (__reduce_max_sync(0xffffffffu, n) + L - 1) / L;
  int nd = 0, all = 0, one = 0;
  SideCounts mine{0, 0};
  // the next parton's loads are in flight while this one is taken in
  int k = kNoLink;
  float2 d = make_float2(-1.0f, -1.0f);
  bool gi = false;
  if (sub < n) {
    k = E.link[E.link_at(0, sub, ev)];
    d = E.dip[dip_at(E, 0, sub, ev)];
    gi = E.flav[E.at(sub, ev)] == kGluon;
  }
#pragma unroll 1
  for (int t = 0; t < rounds; ++t) {
    const int i = t * L + sub, next = i + L;
    const int ck = k;
    const float2 cd = d;
    const bool cg = gi;
    const bool has = i < n && ck != kNoLink && cd.x >= 0.0f;
    // the partner's flavour: from its lane where it was loaded with this one
    const unsigned gluons = __ballot_sync(0xffffffffu, i < n && cg) >> (el * L);
    const bool here = ck >= t * L && ck < (t + 1) * L;
    const bool gk = has && (here ? (gluons >> (ck - t * L) & 1u) != 0u : E.flav[E.at(ck, ev)] == kGluon);
    if (next < n) {
      k = E.link[E.link_at(0, next, ev)];
      d = E.dip[dip_at(E, 0, next, ev)];
      gi = E.flav[E.at(next, ev)] == kGluon;
    }
    const unsigned hm = __ballot_sync(0xffffffffu, has);
    const unsigned g0 = __ballot_sync(0xffffffffu, has && cg), g1 = __ballot_sync(0xffffffffu, has && gk);
    if (has) {
      const int at = nd + __popc(hm & before);
      if (at < kDips) {
        w.dip_x[at][eq] = cd.x;
        w.dip_y[at][eq] = cd.y;
        w.dip_m[at][eq] = static_cast<uint32_t>(i) | (static_cast<uint32_t>(ck) << 8) | (cg ? 1u << 16 : 0u) |
                          (gk ? 1u << 17 : 0u);
        const int sides = 2 * __popc(hm & before), gs = __popc(g0 & before) + __popc(g1 & before);
        int front = all + (combined ? 0 : gs), back = one + sides - (combined ? 0 : gs);
        w.split[cg && !combined ? front++ : 2 * kDips - 1 - back++][eq] = static_cast<uint8_t>(2 * at);
        w.split[gk && !combined ? front : 2 * kDips - 1 - back][eq] = static_cast<uint8_t>(2 * at + 1);
      }
    }
    const int sides = 2 * __popc(hm & group), gs = __popc(g0 & group) + __popc(g1 & group);
    nd += sides / 2;
    all += combined ? 0 : gs;
    one += sides - (combined ? 0 : gs);
    mine.all += sides;
    mine.gluons += gs;
  }
  if (sub == 0 && eq >= 0) {
    w.n_all[eq] = nd <= kDips ? static_cast<uint8_t>(all) : kInRecord;
    w.n_one[eq] = nd <= kDips ? static_cast<uint8_t>(one) : static_cast<uint8_t>(0);
  }
  const int from = lane * L & 31;
  mine.all = __shfl_sync(0xffffffffu, mine.all, from);
  mine.gluons = __shfl_sync(0xffffffffu, mine.gluons, from);
  return mine;
}

// The screens of the warp's events, slot q on each lane (q < 0: none): every
// trial of every event, 32 splitters at a time.  The splitters of the warp's
// events lie one after another (a scan over the lanes' counts), first the
// gluons', then those with one trial; each lane finds the event of its
// splitter from the events' starts in the window of 32.  The partons of
// events whose dipoles did not fit the pool follow, event by event.  An event's smallest bound and the
// smallest of the others are kept by shared-memory minima: each value that
// is not the smallest is displaced or loses exactly once, whatever the order.
// Equal bounds leave the cycle undecided, so which of them is kept is
// immaterial.
template <int kMode>
__device__ __forceinline__ void screen_warp(const DevParams& P0, const DevParams& P, const Events& E, ScreenPool& w,
                                            ScreenResults& r, int q, const EventKey& key, int step) {
  constexpr float kInvCF2 = static_cast<float>(1.0 / (2.0 * kCF));
  constexpr float kInvCA = static_cast<float>(1.0 / kCA);
  constexpr uint32_t kInf = 0x7f800000u;
  const int lane = static_cast<int>(threadIdx.x & 31);
  const unsigned below = lanes_below(lane);
  r.best[lane] = r.second[lane] = kInf;
  const int n_all = q >= 0 ? w.n_all[q] : 0;
  const bool in_record = n_all == kInRecord;
  const uint32_t mine =
      q < 0 || in_record ? 0u : static_cast<uint32_t>(n_all) | (static_cast<uint32_t>(w.n_one[q]) << 16);
  uint32_t incl = mine;  // both kinds' counts in one scan
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  const uint32_t totals = __shfl_sync(0xffffffffu, incl, 31);
  const int gluons = static_cast<int>(totals & 0xffffu), total = gluons + static_cast<int>(totals >> 16);
  // first splitter of the lane's event, of either kind
  const uint32_t starts = incl - mine + (static_cast<uint32_t>(gluons) << 16);
  const int start0 = static_cast<int>(starts & 0xffffu), start1 = static_cast<int>(starts >> 16);
  const bool has0 = (mine & 0xffffu) != 0u, has1 = (mine >> 16) != 0u;
  {  // the lanes with splitters, in the order of their starts
    const unsigned own0 = __ballot_sync(0xffffffffu, has0), own1 = __ballot_sync(0xffffffffu, has1);
    if (has0) w.owner[__popc(own0 & below)] = static_cast<uint8_t>(lane);
    if (has1) w.owner[__popc(own0) + __popc(own1 & below)] = static_cast<uint8_t>(lane);
  }
  unsigned big = __ballot_sync(0xffffffffu, in_record);
  // kernels of a gluon trial by trial, or one trial for all of them
  const int nk_lane = q >= 0 ? (per_dipole<kMode>(P) ? 1 : 1 + P.nf) : 1;
  int base = 0, owners = 0;
  bool from_pool = total > 0;
  __syncwarp();
#pragma unroll 1
  for (;;) {
    int el = 0, i = 0, side = 0, k = 0;
    float x = 0.0f, y = 0.0f;
    bool has = false, gluon = false;
    if (from_pool) {
      const int t = base + lane;
      has = t < total;
      uint32_t mark = has0 && start0 >= base && start0 < base + 32 ? 1u << (start0 - base) : 0u;
      if (has1 && start1 >= base && start1 < base + 32) mark |= 1u << (start1 - base);
      const unsigned marks = __reduce_or_sync(0xffffffffu, mark);
      el = has ? w.owner[owners + __popc(marks & (below | (1u << lane))) - 1] : 0;
      owners += __popc(marks);
      const uint32_t first = __shfl_sync(0xffffffffu, starts, el);
      const int eq = __shfl_sync(0xffffffffu, q, el);
      if (has) {
        const int at = t < gluons ? t - static_cast<int>(first & 0xffffu)
                                  : 2 * kDips - 1 - (t - static_cast<int>(first >> 16));
        const int e = w.split[at][eq];
        const uint32_t m = w.dip_m[e >> 1][eq];
        x = w.dip_x[e >> 1][eq];
        y = w.dip_y[e >> 1][eq];
        side = e & 1;
        i = static_cast<int>((side ? m >> 8 : m) & 255u);
        k = static_cast<int>((side ? m : m >> 8) & 255u);
        gluon = (m >> (16 + side) & 1u) != 0u;
      }
      base += 32;
      if (base >= total) {
        from_pool = false;
        base = 0;
      }
    } else {
      if (big == 0u) break;
      el = __ffs(big) - 1;
      const int n = q >= 0 ? w.n[q] : 0;
      const int at = base + lane;
      if (base >= 2 * __shfl_sync(0xffffffffu, n, el)) {
        big &= big - 1u;
        base = 0;
        continue;
      }
      const int eq = __shfl_sync(0xffffffffu, q, el);
      const int64_t ev = w.ev[eq];
      i = at >> 1;
      side = at & 1;
      if (i < w.n[eq]) {
        k = E.link[E.link_at(side, i, ev)];
        const float2 d = E.dip[dip_at(E, side, i, ev)];
        gluon = E.flav[E.at(i, ev)] == kGluon;
        has = k != kNoLink && d.x >= 0.0f;
        x = d.x;
        y = d.y;
      }
      base += 32;
    }
    EventKey kk;
    kk.id = __shfl_sync(0xffffffffu, key.id, el);
    kk.k0 = kJobKey<kMode> ? __shfl_sync(0xffffffffu, key.k0, el) : 0u;
    kk.k1 = kJobKey<kMode> ? __shfl_sync(0xffffffffu, key.k1, el) : 0u;
    const uint32_t st = static_cast<uint32_t>(__shfl_sync(0xffffffffu, step, el));
    // single-job and keyed launches: the same for every event
    const int nk_event = kJobPhysics<kMode> ? __shfl_sync(0xffffffffu, nk_lane, el) : (per_dipole<kMode>(P0) ? 1 : 1 + P0.nf);
    const int nf = kJobPhysics<kMode> ? __shfl_sync(0xffffffffu, P.nf, el) : P0.nf;
    float h[6], invc = 0.0f;
    U4 r0{0u, 0u, 0u, 0u}, r1 = r0, r2 = r0;
    float h1 = INFINITY, h2 = INFINITY;
    if (has) {
      const uint32_t slot = static_cast<uint32_t>(2 * i + side) * 4u;
      const bool all = gluon && nk_event > 1;
      // 1/c: of a quark, of g -> g g, of a gluon's kernels together (a few ulp)
      invc = !gluon ? x * kInvCF2
                    : (all ? x * kInvCA
                           : __fdividef(1.0f, __fdividef(static_cast<float>(kCA), x) + __fdividef(static_cast<float>(nf), y)));
      r0 = philox_draw<kMode>(P0, kk, st, slot, kDrawTrial);
      h1 = h[0] = trial_bound(r0.x, r0.y, invc);
      if (all) {  // every gluon has at least one g -> q qbar kernel
        r1 = philox_draw<kMode>(P0, kk, st, slot + 1u, kDrawTrial);
        r2 = philox_draw<kMode>(P0, kk, st, slot + 2u, kDrawTrial);
        h[1] = trial_bound(r0.z, r0.w, y);
        h[2] = nk_event > 2 ? trial_bound(r1.x, r1.y, y) : INFINITY;
        h[3] = nk_event > 3 ? trial_bound(r1.z, r1.w, y) : INFINITY;
        h[4] = nk_event > 4 ? trial_bound(r2.x, r2.y, y) : INFINITY;
        h[5] = nk_event > 5 ? trial_bound(r2.z, r2.w, y) : INFINITY;
#pragma unroll
        for (int c = 1; c < 6; ++c) {
          h2 = fminf(h2, fmaxf(h1, h[c]));
          h1 = fminf(h1, h[c]);
        }
      }
      const uint32_t old = atomicMin(&r.best[el], __float_as_uint(h1));
      atomicMin(&r.second[el], min(max(old, __float_as_uint(h1)), __float_as_uint(h2)));
    }
    __syncwarp();
    if (has && r.best[el] == __float_as_uint(h1)) {
      // this splitter's best trial is its event's best so far: its kernel,
      // random words and 1/c
      uint32_t hi = r0.x, lo = r0.y, kappa = 0u;
      if (gluon && nk_event > 1 && h1 != h[0]) {
        invc = y;
        kappa = h1 == h[1] ? 1u : (h1 == h[2] ? 2u : (h1 == h[3] ? 3u : (h1 == h[4] ? 4u : 5u)));
        const bool odd = (kappa & 1u) != 0u;
        const U4 words = kappa == 1u ? r0 : (kappa < 4u ? r1 : r2);
        hi = odd ? words.z : words.x;
        lo = odd ? words.w : words.y;
      }
      r.code[el] = (static_cast<uint32_t>(2 * i + side) << 3) | kappa | (static_cast<uint32_t>(k) << 16) |
                     (gluon ? 1u << 24 : 0u);
      r.hi[el] = hi;
      r.lo[el] = lo;
      r.invc[el] = invc;
    }
    __syncwarp();
  }
}

// Slot states of a pool: empty, live, live with an emission waiting, live
// with its screen's dipoles to be loaded, and four ways to leave: at the
// cutoff, with a full record, at the cycle limit, or at the end of a slice.
// A slot that has left is written back and refilled together with others.
enum : uint8_t {
  kSlotEmpty = 0,
  kSlotLive = 1,
  kSlotPending = 2,
  kSlotLoad = 3,
  kSlotDone = 4,  // and above: the event has left
  kSlotOverflow = 5,
  kSlotLimit = 6,
  kSlotSliced = 7
};

struct WarpPool {
  double lnt[kSlots];
  unsigned long long hash[kSlots];
  ScreenPool sc;
  uint32_t rz_hi[kSlots], rz_lo[kSlots], won[kSlots];  // the waiting emission
  int32_t step[kSlots];
  int32_t first_step[kSlots];    // cycle the event came in at
  int32_t settled_step[kSlots];  // cycle up to which its work counts are in the record
  uint16_t trials[kSlots], dipoles[kSlots];  // per cycle, until its next emission
  uint16_t job[kSlots];
  uint8_t state[kSlots], cyc[kSlots], list[kSlots];
  union {
    ScreenResults r;
    // a warp's share of the block's lists of an emission turn: the waiting
    // events (warp * 64 + slot), the dipoles their emissions move, and those
    // of them with phase space
    struct {
      double q2[kMaxRefresh * 32];
      uint32_t jobs[kMaxRefresh * 32], kept[kMaxRefresh * 32];
      uint16_t tasks[32];
    } m;
  };
};

// What the warps of a block agree on.
struct BlockShared {
  uint32_t vote[2][kMaxThreads / 32];  // running | waiting << 16 of every warp, in turn
  int n_jobs, n_kept;
  double pad;  // the pools behind it stay aligned
};

static_assert(sizeof(BlockShared) + sizeof(WarpPool) * (kMaxThreads / 32) <= 227 * 1024, "16 warps' pools fit an SM");

// Where a launch takes its events from and how far it runs them.  Whole
// batch (kSlice false): events 0 .. E.n - 1 to the cutoff, cursor in counter
// word 6.  Slice (kSlice true): the events of list_in (length *n_in_dev, at
// most n_in), each for at most `cycles` veto cycles; those still active then
// go to list_out (one atomic per warp).
struct SliceArgs {
  const int* list_in;
  const unsigned long long* n_in_dev;
  int64_t n_in;
  unsigned long long* cursor;
  int cycles;
  int* list_out;
  unsigned long long* out_count;
};

// Whether a block (or a warp, at its share) should generate its waiting
// emissions: half of its live events wait, so that the others still fill the
// warps, or flush_at per warp do (a third or a quarter of them was 6 and 13 %
// slower at 10^6 events, two thirds 1 %).
__device__ __forceinline__ bool emission_due(int running, int waiting, int flush_at) {
  return waiting > 0 && (running == 0 || waiting >= flush_at || 2 * waiting >= running + waiting);
}

// Add the work counts of slot q's cycles since its last emission to the
// record.
__device__ __forceinline__ void settle_counts(const Events& E, WarpPool& w, int q) {
  const int cycles = w.step[q] - w.settled_step[q];
  const int ev = w.sc.ev[q];
  atomicAdd(&E.n_trials[ev], cycles * static_cast<int>(w.trials[q]));
  atomicAdd(&E.n_dipoles[ev], cycles * static_cast<int>(w.dipoles[q]));
  w.settled_step[q] = w.step[q];
}

// The event of slot q, which left with `state`, back to the record: its
// scalars, and its status and final scale unless its slice ended.
template <int kMode>
__device__ __forceinline__ void write_back(const DevParams& P0, const Events& E, WarpPool& w, int q, int state) {
  settle_counts(E, w, q);
  const int ev = w.sc.ev[q];
  const double lnt = w.lnt[q];
  E.lnt[ev] = lnt;
  E.hash[ev] = w.hash[q];
  E.n_steps[ev] = w.step[q];
  // every cycle of the stay had a winner but the one that found the cutoff
  atomicAdd(&E.n_winners[ev], w.step[q] - w.first_step[q] - (state == kSlotDone ? 1 : 0));
  if (state == kSlotDone) {
    finish_event(E, ev, GAPS_DONE, job_params<kJobPhysics<kMode>>(P0, E, w.job[q]).tc);
  } else if (state != kSlotSliced) {
    finish_early(E, ev, state == kSlotLimit ? GAPS_STEP_LIMIT : GAPS_OVERFLOW, lnt);
    if (state == kSlotLimit) atomicAdd(&E.counters[1], 1ull);
  }
}

template <int kMode, bool kSlice>
__global__ void __launch_bounds__(kMaxThreads)
    k_shower_persistent(DevParams P0, Events E, int flush_at, SliceArgs sl) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  BlockShared& blk = *reinterpret_cast<BlockShared*>(s_raw);
  WarpPool* const pools = reinterpret_cast<WarpPool*>(s_raw + sizeof(BlockShared));
  const int tid = static_cast<int>(threadIdx.x), warp = tid >> 5, n_warps = static_cast<int>(blockDim.x >> 5);
  WarpPool& w = pools[warp];
  const int lane = static_cast<int>(threadIdx.x & 31);
  const unsigned below = lanes_below(lane);
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
  unsigned long long* cursor = kSlice ? sl.cursor : &E.counters[6];
  const int64_t total = kSlice ? (sl.n_in_dev ? min(sl.n_in, static_cast<int64_t>(*sl.n_in_dev)) : sl.n_in) : E.n;
  int64_t left = total;  // events the cursor had not handed out when this warp last looked
  int vote = 0;
  bool ended = false;     // no event left, here or at the cursor
  bool refilled = false;  // in the last turn: run what came in before asking again
  w.state[lane] = w.state[lane + 32] = kSlotEmpty;
  __syncwarp();
  unsigned turn = 0;
#pragma unroll 1
  for (;;) {
    // The pool: which slots can run, wait for their emission, are free.
    int s0 = w.state[lane], s1 = w.state[lane + 32];
    unsigned run0 = __ballot_sync(0xffffffffu, s0 == kSlotLive), run1 = __ballot_sync(0xffffffffu, s1 == kSlotLive);
    unsigned wait0 = __ballot_sync(0xffffffffu, s0 == kSlotPending);
    unsigned wait1 = __ballot_sync(0xffffffffu, s1 == kSlotPending);
    int running = __popc(run0) + __popc(run1), waiting = __popc(wait0) + __popc(wait1);
    const int free = kSlots - running - waiting;
    bool load = false;  // events came in or emitted: their dipoles for the screen
    if (free == kSlots ? !ended : free >= kSlots / 4 && left > 0 && !refilled) {
      // Write the events that have left back, and refill their slots from
      // the global cursor: an even share of what is left at first (small
      // batches spread over every warp), and no more than a fraction of it
      // near the end, so that the warps end together.
      unsigned long long base = 0;
      int take = 0;
      if (left > 0) {
        // (in single precision: any share near the even one will do)
        float share = ceilf(__fdividef(static_cast<float>(left), static_cast<float>(warps)));
        if (left < total) share = ceilf(0.5f * share);
        const int want = min(free, max(1, static_cast<int>(fminf(share, 64.0f))));
        if (lane == 0) base = atomicAdd(cursor, static_cast<unsigned long long>(want));
        base = __shfl_sync(0xffffffffu, base, 0);
        const int64_t have = total - static_cast<int64_t>(base);
        left = have - want;
        take = have <= 0 ? 0 : static_cast<int>(min(have, static_cast<int64_t>(want)));
      }
      int given = 0;
#pragma unroll 1
      for (int o = 0; o < 2; ++o) {
        const int q = lane + 32 * o, state = o ? s1 : s0;
        const bool out = state >= kSlotDone, done = out && state != kSlotSliced;
        if (out) write_back<kMode>(P0, E, w, q, state);
        const unsigned dm = __ballot_sync(0xffffffffu, done);
        if (dm != 0u && lane == 0) atomicAdd(&E.counters[0], static_cast<unsigned long long>(__popc(dm)));
        count_job_done(E, out ? w.sc.ev[q] : 0, done);
        if constexpr (kSlice) {
          const bool sliced = state == kSlotSliced;
          const unsigned sm = __ballot_sync(0xffffffffu, sliced);
          if (sm != 0u) {
            unsigned long long at = 0;
            if (lane == 0) at = atomicAdd(sl.out_count, static_cast<unsigned long long>(__popc(sm)));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (sliced) sl.list_out[at + __popc(sm & below)] = w.sc.ev[q];
          }
        }
        const bool open = out || state == kSlotEmpty;
        const unsigned om = __ballot_sync(0xffffffffu, open);
        const int r = given + __popc(om & below);
        given += __popc(om);
        if (open && r < take) {
          const int64_t at = static_cast<int64_t>(base) + r;
          const int ev = kSlice && sl.list_in ? sl.list_in[at] : static_cast<int>(at);
          w.sc.ev[q] = ev;
          w.job[q] = kJobKey<kMode> ? E.job_of[ev] : static_cast<uint16_t>(0);
          w.sc.n[q] = static_cast<uint8_t>(E.n_partons[ev]);
          w.step[q] = w.first_step[q] = w.settled_step[q] = E.n_steps[ev];
          w.lnt[q] = E.lnt[ev];
          w.hash[q] = E.hash[ev];
          w.cyc[q] = 0;
        }
        if (open) w.state[q] = r < take ? kSlotLoad : kSlotEmpty;
      }
      ended = free == kSlots && take == 0;
      refilled = true;
      running += take;
      load = true;
    } else {
      refilled = false;
    }
    // The warps of a block generate their emissions together: packed into as
    // few warps as hold them, and with their code coming through the
    // instruction cache once.  (The block lives while one of its warps has
    // events.)
    if (lane == 0) blk.vote[vote][warp] = static_cast<uint32_t>(running) | (static_cast<uint32_t>(waiting) << 16);
    if (tid == 0) blk.n_jobs = blk.n_kept = 0;
    const bool all_ended = __syncthreads_and(ended) != 0;
    uint32_t sum = 0u, before = 0u;
    for (int k = 0; k < n_warps; ++k) {
      const uint32_t v = blk.vote[vote][k];
      sum += v;
      before += k < warp ? v >> 16 : 0u;
    }
    vote ^= 1;
    if (all_ended) break;
    const int all_waiting = static_cast<int>(sum >> 16);
    if (emission_due(static_cast<int>(sum & 0xffffu), all_waiting, flush_at * n_warps)) {
      // GenerateEmission for the waiting events, one per thread, then the
      // dipoles they moved, spread over the block: first their masses, then
      // the entries of those with phase space (about half of them).
      const int r0 = static_cast<int>(before) + __popc(wait0 & below);
      const int r1 = static_cast<int>(before) + __popc(wait0) + __popc(wait1 & below);
      const int tasks = min(all_waiting, n_warps * 32);  // the first ones; the others keep waiting
      if (s0 == kSlotPending && r0 < tasks) pools[r0 >> 5].m.tasks[r0 & 31] = static_cast<uint16_t>(warp * kSlots + lane);
      if (s1 == kSlotPending && r1 < tasks)
        pools[r1 >> 5].m.tasks[r1 & 31] = static_cast<uint16_t>(warp * kSlots + lane + 32);
      __syncthreads();
      // Four lanes a task while the tasks then take at most a warp on each of
      // the SM's schedulers, whose FP64 issue one warp fills: a chain of 90
      // FP64 instructions instead of 161.  Beyond, a thread a task takes half
      // the instructions.  100 events 0.197 -> 0.190 ms, 2x10^4 0.253 ->
      // 0.244 (up to 1, 2, 4 or 8 such warps alike), 10^6 unchanged.
      const bool quads = tasks <= 8 * min(n_warps, kSchedulers);
      // the task of this lane, or the last one on the lanes left over
      const int at_task = quads ? tid >> 2 : tid;
      const bool has = at_task < tasks;
      if (quads ? warp * 8 < tasks : has) {
        const int r = min(at_task, tasks - 1);
        const int task = pools[r >> 5].m.tasks[r & 31], q = task & (kSlots - 1);
        WarpPool& o = pools[task >> 6];
        const uint32_t won = o.won[q];
        const int64_t ev = o.sc.ev[q];
        EmitTask t;
        t.ev = static_cast<int32_t>(ev);
        t.i = static_cast<uint8_t>(won & 255u);
        t.k = static_cast<uint8_t>((won >> 8) & 255u);
        t.side = static_cast<uint8_t>((won >> 16) & 15u);
        t.kappa = static_cast<uint8_t>((won >> 20) & 15u);
        t.kind = static_cast<uint8_t>(won >> 24);
        t.n = o.sc.n[q];
        t.step = o.step[q] - 1;
        t.lnt = o.lnt[q];
        t.rz_hi = o.rz_hi[q];
        t.rz_lo = o.rz_lo[q];
        const DipoleRecord rec = E.drec[E.at(t.side == 0 ? t.i : t.k, ev)];
        t.q2 = rec.q2;
        t.zp = rec.zp;
        t.ls = rec.ls;
        const auto reserve = [&](int count) { return atomicAdd(&blk.n_jobs, count); };
        const auto put = [&](int at, uint32_t job) { pools[at >> 7].m.jobs[at & 127] = job; };
        if (quads)
          emit_warp4<kMode>(P0, E, t, has, reserve, put, r);
        else
          cycle_emit<kMode>(P0, E, t, reserve, put, r);
        if (has && (!quads || (tid & 3) == 0)) {
          settle_counts(E, o, q);
          o.sc.n[q] = static_cast<uint8_t>(t.n + 1);
          bool over = false;
          if constexpr (kSlice) over = o.cyc[q] >= sl.cycles;
          o.state[q] = over ? kSlotSliced : kSlotLoad;
        }
      }
      __syncthreads();
      const int jobs = blk.n_jobs;
#pragma unroll 1
      for (int j0 = warp * 32; j0 < jobs; j0 += n_warps * 32) {
        const int j = j0 + lane;
        bool keep = false;
        uint32_t job = 0u;
        double q2 = 0.0;
        if (j < jobs) {
          job = pools[j >> 7].m.jobs[j & 127];
          const int task = pools[refresh_task(job) >> 5].m.tasks[refresh_task(job) & 31];
          const WarpPool& o = pools[task >> 6];
          const int64_t ev = o.sc.ev[task & (kSlots - 1)];
          q2 = refresh_mass(E, ev, job);
          keep = has_phase_space(job_params<kJobPhysics<kMode>>(P0, E, o.job[task & (kSlots - 1)]), q2);
          if (!keep) refresh_store(E, ev, job, no_dipole(q2));
        }
        const unsigned km = __ballot_sync(0xffffffffu, keep);
        int at = 0;
        if (lane == 0 && km != 0u) at = atomicAdd(&blk.n_kept, __popc(km));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(km & below);
        if (keep) {
          pools[at >> 7].m.kept[at & 127] = job;
          pools[at >> 7].m.q2[at & 127] = q2;
        }
      }
      __syncthreads();
      const int kept = blk.n_kept;
#pragma unroll 1
      for (int j = tid; j < kept; j += n_warps * 32) {
        const uint32_t job = pools[j >> 7].m.kept[j & 127];
        const int task = pools[refresh_task(job) >> 5].m.tasks[refresh_task(job) & 31];
        const WarpPool& o = pools[task >> 6];
        refresh_store(E, o.sc.ev[task & (kSlots - 1)], job,
                      make_dipole(job_params<kJobPhysics<kMode>>(P0, E, o.job[task & (kSlots - 1)]),
                                  pools[j >> 7].m.q2[j & 127]));
      }
      __syncthreads();
      load = true;
    }
    if (load) {
      __syncwarp();
      s0 = w.state[lane];
      s1 = w.state[lane + 32];
      const unsigned l0 = __ballot_sync(0xffffffffu, s0 == kSlotLoad), l1 = __ballot_sync(0xffffffffu, s1 == kSlotLoad);
      if (s0 == kSlotLoad) w.list[__popc(l0 & below)] = static_cast<uint8_t>(lane);
      if (s1 == kSlotLoad) w.list[__popc(l0) + __popc(l1 & below)] = static_cast<uint8_t>(lane + 32);
      __syncwarp();
      const int count = __popc(l0) + __popc(l1);
#pragma unroll 1
      for (int k0 = 0; k0 < count; k0 += 32) {
        const int q = k0 + lane < count ? w.list[k0 + lane] : -1;
        const SideCounts sides =
            load_dipoles<kMode>(P0, E, w.sc, q, q >= 0 ? w.job[q] : 0, lanes_each(min(count - k0, 32)));
        if (q >= 0) {
          const DevParams& P = job_params<kJobPhysics<kMode>>(P0, E, w.job[q]);
          w.trials[q] = static_cast<uint16_t>(sides.all + sides.gluons * (per_dipole<kMode>(P) ? 0 : P.nf));
          w.dipoles[q] = static_cast<uint16_t>(sides.all);
          w.state[q] = kSlotLive;
        }
      }
      __syncwarp();
    }
    // A few veto cycles of up to 32 events each, the halves of the pool first
    // in turn.
#pragma unroll 1
    for (int c = 0; c < kTurns; ++c) {
      s0 = w.state[lane];
      s1 = w.state[lane + 32];
      run0 = __ballot_sync(0xffffffffu, s0 == kSlotLive);
      run1 = __ballot_sync(0xffffffffu, s1 == kSlotLive);
      running = __popc(run0) + __popc(run1);
      waiting = __popc(__ballot_sync(0xffffffffu, s0 == kSlotPending)) + __popc(__ballot_sync(0xffffffffu, s1 == kSlotPending));
      if (running == 0 || (c > 0 && emission_due(running, waiting, flush_at))) break;
      const bool swap = (++turn & 1u) != 0u;
      if (s0 == kSlotLive) w.list[__popc(run0 & below) + (swap ? __popc(run1) : 0)] = static_cast<uint8_t>(lane);
      if (s1 == kSlotLive) w.list[__popc(run1 & below) + (swap ? 0 : __popc(run0))] = static_cast<uint8_t>(lane + 32);
      __syncwarp();
      const int q = lane < running ? w.list[lane] : -1;
      const int64_t ev = q >= 0 ? w.sc.ev[q] : -1;
      const int job = q >= 0 ? w.job[q] : 0;
      const DevParams& P = job_params<kJobPhysics<kMode>>(P0, E, job);
      const int step = q >= 0 ? w.step[q] : 0;
      const bool limited = q >= 0 && step >= P.max_steps;
      EventKey key{0u, 0u, 0u};
      if (q >= 0) key = event_key<kMode>(P, E, ev, job);
      screen_warp<kMode>(P0, P, E, w.sc, w.r, limited ? -1 : q, key, step);
      const bool lead = q >= 0 && !limited;
      int verdict = kScreenNone;
      double lnt = 0.0;
      EmitTask task;
      if (lead) {
        lnt = w.lnt[q];
        const uint32_t best = w.r.best[lane], code = w.r.code[lane];
        verdict = screen_verdict<kMode>(P, E, ev, lnt, __uint_as_float(best), __uint_as_float(w.r.second[lane]),
                                        w.r.invc[lane], best == 0x7f800000u ? -1 : static_cast<int>(code & 4095u),
                                        code >> 16, w.r.hi[lane], w.r.lo[lane], task);
        if (verdict == kScreenUndecided) atomicAdd(&E.counters[2], 1ull);  // full FP64 cycle
      }
      bool have = verdict == kScreenWinner;
      // The exact selection's results in their own variables: the call, out of
      // line, takes them by address, and `task` itself would live in local
      // memory for every cycle (10^6 events 5.55 -> 5.33 ms; the plain step,
      // at half the registers, is 2 % faster with it there).
      if (__any_sync(0xffffffffu, verdict == kScreenUndecided)) {
        EmitTask exact;
        bool found = false;
        fallback_warp<kMode>(P0, E, verdict == kScreenUndecided, ev, job, key, step, q >= 0 ? w.sc.n[q] : 0, lnt, found,
                             exact);
        if (verdict == kScreenUndecided) {
          have = found;
          task = exact;
        }
      }
      if (limited) w.state[q] = kSlotLimit;
      if (lead) {
        w.step[q] = step + 1;
        uint8_t state = kSlotDone;  // CheckCutoff
        if (have) {
          unsigned long long hash = w.hash[q];
          w.lnt[q] = task.lnt;
          const bool accept = accept_or_veto<kMode>(P, E, key, step, task, hash);
          w.hash[q] = hash;
          state = kSlotLive;
          if (accept) {
            w.rz_hi[q] = task.rz_hi;
            w.rz_lo[q] = task.rz_lo;
            w.won[q] = static_cast<uint32_t>(task.i) | (static_cast<uint32_t>(task.k) << 8) |
                       (static_cast<uint32_t>(task.side) << 16) | (static_cast<uint32_t>(task.kappa) << 20) |
                       (static_cast<uint32_t>(task.kind) << 24);
            state = w.sc.n[q] >= E.cap ? kSlotOverflow : kSlotPending;
          }
          if constexpr (kSlice) {
            const int cyc = w.cyc[q] + 1;
            w.cyc[q] = static_cast<uint8_t>(cyc);
            if (state == kSlotLive && cyc >= sl.cycles) state = kSlotSliced;
          }
        }
        w.state[q] = state;
      }
      __syncwarp();
    }
  }
}

template <int kMode, bool kSlice>
cudaError_t launch_m(const DevParams& P, const Events& E, const gaps_persistent_config& cfg, const SliceArgs& sl,
                     cudaStream_t s) {
  const int64_t n = kSlice ? sl.n_in : E.n;
  int dev = 0, sms = 0, fit = 0;
  int threads = cfg.block_threads;
  if (threads != 64 && threads != 128 && threads != 256 && threads != 512) return cudaErrorInvalidValue;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // Batches with fewer events than the device has warps: one warp per block,
  // so that they spread over the SMs.
  if (n <= static_cast<int64_t>(sms) * (kMaxThreads / 32)) threads = 32;
  const size_t smem = sizeof(BlockShared) + sizeof(WarpPool) * static_cast<size_t>(threads / 32);
  auto* kernel = k_shower_persistent<kMode, kSlice>;
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(sizeof(BlockShared) + sizeof(WarpPool) * (kMaxThreads / 32)));
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kernel, threads, smem);
  if (e != cudaSuccess) return e;
  if (fit < 1) return cudaErrorInvalidConfiguration;
  const int per_sm = cfg.blocks_per_sm > 0 && cfg.blocks_per_sm < fit ? cfg.blocks_per_sm : fit;
  // At least a dozen events per warp while there are fewer than fill the
  // device: the emissions then fill their warps better (six, eight or sixteen
  // a warp measure within 3 % from 3x10^3 to 5x10^4 events).
  const int64_t warps = threads == 32 ? n : (n + 11) / 12;
  const int64_t blocks = std::min(static_cast<int64_t>(sms) * per_sm,
                                  std::max<int64_t>((warps + threads / 32 - 1) / (threads / 32), std::min<int64_t>(sms, n)));
  if (blocks == 0) return cudaSuccess;
  kernel<<<static_cast<unsigned>(blocks), threads, smem, s>>>(P, E, emissions_awaited(cfg.compact_period), sl);
  return cudaGetLastError();
}

template <bool kSlice>
cudaError_t launch_shape(const DevParams& P, const Events& E, const gaps_persistent_config& cfg, const SliceArgs& sl,
                         cudaStream_t s) {
  switch (launch_mode(P, E)) {
    case kModeKeyed:
      if constexpr (kSlice) return launch_m<kModeKeyed, kSlice>(P, E, cfg, sl, s);
      return launch_m<kModeMulti, kSlice>(P, E, cfg, sl, s);  // the job table holds the same parameters
    case kModeKeyedDipole:
      if constexpr (kSlice) return launch_m<kModeKeyedDipole, kSlice>(P, E, cfg, sl, s);
      return launch_m<kModeMulti, kSlice>(P, E, cfg, sl, s);
    case kModeMulti: return launch_m<kModeMulti, kSlice>(P, E, cfg, sl, s);
    case kModeSingleDipole: return launch_m<kModeSingleDipole, kSlice>(P, E, cfg, sl, s);
    default: return launch_m<kModeSingleKernel, kSlice>(P, E, cfg, sl, s);
  }
}

}  // namespace

cudaError_t launch_shower_persistent(const DevParams& P, const Events& E, const gaps_persistent_config& cfg,
                                     cudaStream_t s) {
  if (E.n == 0) return cudaSuccess;
  return launch_shape<false>(P, E, cfg, SliceArgs{}, s);
}

cudaError_t launch_shower_slice(const DevParams& P, const Events& E, const gaps_persistent_config& cfg,
                                const int* list_in, int64_t n_in, const unsigned long long* n_in_dev,
                                unsigned long long* cursor, int cycles, int* list_out, unsigned long long* out_count,
                                cudaStream_t s) {
  if (n_in == 0 || cycles < 1 || cycles > 255) return n_in == 0 ? cudaSuccess : cudaErrorInvalidValue;
  const SliceArgs sl{list_in, n_in_dev, n_in, cursor, cycles, list_out, out_count};
  return launch_shape<true>(P, E, cfg, sl, s);
}

}  // namespace gaps

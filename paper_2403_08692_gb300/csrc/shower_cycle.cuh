// One veto cycle of one event (Sec. 2, App. A, App. C), split in two phases
// and shared by every shower form:
//   cycle_select_veto  SelectWinnerEmission + CheckCutoff + AcceptOrVeto
//   cycle_emit         GenerateEmission for an accepted winner
// The caller runs the first phase for a dense set of active events, queues
// the accepted ones (about one in ten) and runs the second phase on the
// queue, so the FP64-heavy splitting never executes in a warp whose other
// lanes idle.
//
// GB300 runs FP64 at about 1/74 of its FP32 rate, so the cycle spends FP64
// only where the result must be FP64:
//  * Trial screening.  Every trial's scale is ranked by its key
//    log2(t'/t) = log2(r) / c in FP32, from a per-dipole cache of 1/c; each
//    key carries a bound on its FP32 error.  When one trial's key beats every
//    other trial's and the cutoff by more than the bounds, it is the winner
//    the exact FP64 comparison would pick, and only its scale is evaluated in
//    FP64.  Otherwise (about 1e-4 of cycles) the whole cycle is redone with
//    every trial in FP64, exactly as the oracle does it.
//  * Log-space evolution.  The event carries L = ln t; a winner moves it to
//    L + ln(r)/c (Eq. A.6 in logarithms), so a cycle needs one FP64 log and
//    no exp; t itself is formed only for an accepted emission.
//  * Veto.  z, y and the acceptance ratio are formed in FP32 with an error
//    bound; only a veto number within the bound of the ratio is decided in
//    FP64.  z and y are recomputed in FP64 for the accepted emissions.
//  * Dipole cache.  A dipole's trial density depends only on its invariant
//    mass, which changes only when an emission moves one of its partons, so
//    Q^2, z+, ln(z+/z-) and its inverse (FP64) and 1/c (FP32) are stored per dipole and
//    recomputed once per dipole an emission touches.
#pragma once
#include "gaps_device.cuh"

namespace gaps {

// Error allowances of the FP32 screens, several times the worst-case error of
// the FP32 operations involved.  Trial key = log2(r) * (1/c): the 24-bit
// uniform is within 2^-22 relative of r (3.4e-7 absolute in log2 r), MUFU
// log2 adds at most 2e-6 (1 + |log2 r|), the cached 1/c is within 1e-6
// relative, the product rounds once; so |key error| <= 2e-6/c + 7e-6 |key|,
// allowed as 4e-6/c + 1.6e-5 |key|.  Veto ratio: z, 1 - z and y from MUFU
// exp/log and ~20 FP32 operations carry <= 1e-5 relative error and (1 - y)
// <= 5e-6 absolute, allowed as 5e-5 (ratio + r) + 2e-5.
constexpr float kKeyRelInvc = 4e-6f;
constexpr float kKeyRelKey = 1.6e-5f;
constexpr float kVetoRel = 5e-5f;
constexpr float kVetoAbs = 2e-5f;

__device__ __forceinline__ V4 load_p(const Events& E, int slot, int64_t ev) {
  const size_t a = E.at(slot, ev);
  return V4{E.e[a], E.px[a], E.py[a], E.pz[a]};
}
__device__ __forceinline__ void store_p(const Events& E, int slot, int64_t ev, const V4& p) {
  const size_t a = E.at(slot, ev);
  E.e[a] = p.e;
  E.px[a] = p.x;
  E.py[a] = p.y;
  E.pz[a] = p.z;
}

__device__ __forceinline__ size_t dip_at(const Events& E, int side, int slot, int64_t ev) {
  return E.link_at(side, slot, ev);
}

// Cache entry of a dipole of invariant mass q2: FP64 Q^2, z+ = (1 + b)/2
// with b = sqrt(1 - 4 t_C/Q^2) (the oracle's formula) and 1/ln(z+/z-) with
// z- = 1 - z+, and the FP32 screen entry x = 1/(a ln(z+/z-)), y = 1/(a T_R/2
// (z+ - z-)), a = alpha_s^over/(2 pi).  x = -1 marks a dipole without phase
// space (Q^2 < 4 t_C, the oracle's FP64 test).  z+/z- = (1 + b)/(1 - b)
// equals (1 + b)^2 Q^2 / (4 t_C) since 1 - b^2 = 4 t_C/Q^2: no division, and
// none of the cancellation in 1 - z+ (the values agree with the oracle's two
// logarithms to about 1e-13 relative at LEP energies).
struct DipoleEntry {
  DipoleRecord rec;
  float2 screen;
};

// Whether a dipole of mass squared q2 has phase space: not Q^2 < 4 t_C, the
// sign of their difference (exact where they are close) read from its bits.
__device__ __forceinline__ bool has_phase_space(const DevParams& P, double q2) {
  return __double_as_longlong(q2 - 4.0 * P.tc) >= 0;
}
// The entry of a dipole without.
__device__ __forceinline__ DipoleEntry no_dipole(double q2) {
  DipoleEntry d;
  d.rec.q2 = q2;
  d.rec.zp = d.rec.inv_ls = d.rec.ls = 0.0;
  d.screen = make_float2(-1.0f, -1.0f);
  return d;
}

__device__ __forceinline__ DipoleEntry make_dipole(const DevParams& P, double q2) {
  if (!has_phase_space(P, q2)) return no_dipole(q2);
  DipoleEntry d;
  d.rec.q2 = q2;
  // b = sqrt(1 - 4 t_C/Q^2) = a / sqrt(Q^2 a) with a = Q^2 - 4 t_C: one
  // reciprocal square root instead of a division and a square root
  const double a = q2 - 4.0 * P.tc;
  const double b = __double_as_longlong(a) > 0 ? a * rsqrt_fp64(q2 * a) : 0.0;
  const double b1 = 1.0 + b;
  d.rec.zp = 0.5 * b1;
  const double ls = log_fp64((b1 * b1) * (q2 * P.inv_4tc));
  d.rec.ls = ls;
  d.rec.inv_ls = rcp_fp64(ls);
  d.screen = make_float2(__fdividef(1.0f, P.as2pi_f * f32_from_f64(ls)),
                         __fdividef(1.0f, P.as2pi_f * 0.5f * static_cast<float>(kTR) * f32_from_f64(b)));
  return d;
}

// The entry of the dipole between slots x and k, partners on x's side `side`:
// its screen entry on both sides, its record at the colour end.
__device__ __forceinline__ void store_dipole(const Events& E, int64_t ev, int x, int side, int k,
                                             const DipoleEntry& d) {
  E.dip[dip_at(E, side, x, ev)] = d.screen;
  E.dip[dip_at(E, 1 - side, k, ev)] = d.screen;
  if (d.screen.x < 0.0f) return;
  E.drec[E.at(side == 0 ? x : k, ev)] = d.rec;
}

// 32-bit float close to the 52-bit uniform built from (hi, lo): relative
// error below 2^-22 for every value.
__device__ __forceinline__ float unit_float(uint32_t hi, uint32_t lo) {
  const float a = __uint2float_rn(hi >> 6);
  const float b = __uint2float_rn(lo >> 6);
  return fmaf(a, 0x1p-26f, fmaf(b, 0x1p-52f, 0x1p-53f));
}


// A dipole whose cache entry an emission invalidated: parton slots x and k,
// partners on x's side `side`, of the event of task t in the block's queue.
// An emission invalidates at most kMaxRefresh dipoles: (i, j), (j, k) and
// the other partners of the splitter and of the spectator.
constexpr int kMaxRefresh = 4;
__device__ __forceinline__ uint32_t pack_refresh(int t, int x, int side, int k) {
  return static_cast<uint32_t>(t) | (static_cast<uint32_t>(x) << 10) | (static_cast<uint32_t>(k) << 18) |
         (static_cast<uint32_t>(side) << 26);
}

// 1/c of a kernel for a dipole, c = alpha_s^over/(2 pi) * integral of
// P^over over [z-, z+].
__device__ __forceinline__ double inv_c_fp64(const DevParams& P, int kind, double zp, double inv_ls) {
  if (kind == kGtoQQ) return rcp_fp64(P.as2pi_qq * (zp - (1.0 - zp)));
  return inv_ls * (kind == kQtoQG ? P.inv_as2pi_2cf : P.inv_as2pi_ca);
}

// 1/c of a gluon's kernels together (the per-dipole trial): c summed over
// the kernels in their order, as the oracle sums it.
__device__ __forceinline__ double inv_c_sum_fp64(const DevParams& P, double zp, double ls) {
  const double c_gg = ls * P.as2pi_ca;
  const double c_qq = P.as2pi_qq * (zp - (1.0 - zp));
  double c = c_gg;
#pragma unroll 1
  for (int f = 0; f < P.nf; ++f) c += c_qq;
  return rcp_fp64(c);
}

// The kernel of a winning gluon dipole in the per-dipole mode: kappa with
// probability c_kappa / c_sum, by the running sum against v c_sum.
__device__ __forceinline__ int choose_kernel(const DevParams& P, double zp, double ls, double v) {
  const double c_gg = ls * P.as2pi_ca;
  const double c_qq = P.as2pi_qq * (zp - (1.0 - zp));
  double c_sum = c_gg;
#pragma unroll 1
  for (int f = 0; f < P.nf; ++f) c_sum += c_qq;
  const double target = v * c_sum;
  double cum = c_gg;
  if (target < cum) return 0;
#pragma unroll 1
  for (int q = 1; q <= P.nf; ++q) {
    cum += c_qq;
    if (target < cum) return q;
  }
  return P.nf;
}

// The full FP64 SelectWinnerEmission (every trial exact, from the dipole
// records); the fallback of the FP32 screen.  The log-space scale of trial
// j is L + ln(r_j)/c_j; the highest above ln t_C wins, the first on ties.
// This form covers partons first, first + stride, ... and keeps, in *best,
// *code and w, the best of those trials above the incoming *best (the first
// in loop order on ties; code = (2 i + side) * 8 + kappa orders the trials
// as the loop does); returns whether one was found.
template <int kMode>
__device__ inline bool select_winner_fp64_range(const DevParams& P, const Events& E, int64_t ev, const EventKey& key,
                                                int step, int n, double lnt, int first, int stride, EmitTask& w,
                                                double& best, int& code) {
  bool found = false;
  for (int i = first; i < n; i += stride) {
    const bool gluon = E.flav[E.at(i, ev)] == kGluon;
    const bool combined = gluon && per_dipole<kMode>(P);
    const int nk = gluon && !combined ? 1 + P.nf : 1;
    for (int side = 0; side < 2; ++side) {
      const int k = E.link[E.link_at(side, i, ev)];
      if (k == kNoLink || E.dip[dip_at(E, side, i, ev)].x < 0.0f) continue;
      const DipoleRecord rec = E.drec[E.at(side == 0 ? i : k, ev)];
      for (int kp = 0; kp < nk; kp += 2) {
        const U4 r = philox_draw<kMode>(P, key, static_cast<uint32_t>(step),
                                        static_cast<uint32_t>((2 * i + side) * 4 + kp / 2), kDrawTrial);
        for (int h = 0; h < 2 && kp + h < nk; ++h) {
          const int kappa = kp + h;
          const int kind = combined ? kKindUnchosen : (gluon ? (kappa == 0 ? kGtoGG : kGtoQQ) : kQtoQG);
          const double u = h ? to_unit(r.z, r.w) : to_unit(r.x, r.y);
          const double inv_c =
              combined ? inv_c_sum_fp64(P, rec.zp, rec.ls) : inv_c_fp64(P, kind, rec.zp, rec.inv_ls);
          const double lt = fma(log_fp64(u), inv_c, lnt);
          if (lt > best) {
            best = lt;
            code = (2 * i + side) * 8 + kappa;
            found = true;
            w.lnt = lt;
            w.q2 = rec.q2;
            w.zp = rec.zp;
            w.ls = rec.ls;
            w.i = i;
            w.k = k;
            w.side = side;
            w.kappa = kappa;
            w.kind = kind;
          }
        }
      }
    }
  }
  return found;
}

// The serial form: every parton in one thread.  Returns false if no trial
// is above t_C.
template <int kMode>
__device__ inline bool select_winner_fp64(const DevParams& P, const Events& E, int64_t ev, const EventKey& key, int step,
                                   int n, double lnt, EmitTask& w) {
  double best = P.ln_tc;
  int code = 0;
  return select_winner_fp64_range<kMode>(P, E, ev, key, step, n, lnt, 0, 1, w, best, code);
}

// Exact FP64 acceptance ratio of Eq. (A.9) with the (1 - y) factor, for a
// given z.  Returns -1 when y >= 1.
__device__ __forceinline__ double veto_ratio_fp64(const DevParams& P, int kind, double t, double q2, double z) {
  const double y = t / (q2 * z * (1.0 - z));
  if (!(y < 1.0)) return -1.0;
  const double f = (1.0 - y) * alpha_s(P, t) * kernel_p(kind, z, y);
  const double g = P.as_over * kernel_over(kind, z);
  return f / g;
}

// z from Eq. (A.8) in FP64, in a cancellation-free form: for the 1/(1-z)
// kernels 1 - z = z+ (z-/z+)^r, i.e. z = z- - z+ expm1(-r ln(z+/z-)).
__device__ __forceinline__ double z_fp64(int kind, double zp, double lsoft, double r) {
  const double zm = 1.0 - zp;
  if (kind == kGtoQQ) return fma(zp - zm, r, zm);
  return fma(-zp, expm1_neg_fp64(-r * lsoft), zm);
}

// The veto decided in FP64 (a veto number within the FP32 ratio's error of
// it, about one cycle in 10^4): out of line, its logarithm, exponentials and
// divisions would make up much of the cycle's code.
static __device__ __noinline__ bool accept_fp64(const DevParams& P, int kind, double lnt, double q2, double zp, double ls,
                                                double rz, double rv) {
  const double z = z_fp64(kind, zp, ls, rz);
  const double ratio = veto_ratio_fp64(P, kind, exp_fp64(lnt), q2, z);
  return ratio >= 0.0 && rv < ratio;
}

enum : int { kCycleVetoed = 0, kCycleFinished = 1, kCycleAccepted = 2 };

// The serving pool counts every job's finished events (E.job_done, set only
// for the pool): the lanes of a warp that finished events of the same job
// add them with one atomic.  Every lane of the warp must call it.
__device__ __forceinline__ void count_job_done(const Events& E, int64_t ev, bool finished) {
  if (!E.job_done) return;  // the same for every lane (a launch argument)
  const int job = finished ? static_cast<int>(E.job_of[ev]) : -1;
  const unsigned peers = __match_any_sync(0xffffffffu, job);
  if (finished && static_cast<int>(threadIdx.x & 31) == __ffs(peers) - 1)
    atomicAdd(&E.job_done[job], static_cast<unsigned long long>(__popc(peers)));
}

// Leave the active state with `status`, recording the final scale.
__device__ __forceinline__ void finish_event(const Events& E, int64_t ev, int status, double t) {
  E.status[ev] = status;
  E.t[ev] = t;
}

// The same before the cutoff (a full record, the cycle limit), at ln t = lnt:
// rare, so out of line.
static __device__ __noinline__ void finish_early(const Events& E, int64_t ev, int status, double lnt) {
  finish_event(E, ev, status, exp_fp64(lnt));
}

// The |key| bound of a trial, h = |key| - m >= 0 with key = log2(u)/c <= 0
// and m its error allowance: its upper bound, negated, so
// that positive floats order as their bits.  u >= 2^-53: no denormals.
__device__ __forceinline__ float trial_bound(uint32_t hi, uint32_t lo, float invc) {
  float lg;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(lg) : "f"(unit_float(hi, lo)));
  return fmaxf(invc * fmaf(-lg, 1.0f - kKeyRelKey, -kKeyRelInvc), 0.0f);
}

// The FP32 screen of SelectWinnerEmission over the trials of partons
// first, first + stride, ... of an event: the smallest |key| bound (h1) with
// its 1/c, trial and random words, the smallest bound of every other trial,
// and the work counts.  Equal smallest bounds leave the cycle undecided, so
// which trial is kept is immaterial.
struct Screen {
  float h1, h2, invc;
  int best_code;  // (2 i + side) * 8 + kappa, -1: no trial
  uint32_t best_hi, best_lo;
  uint32_t best_aux;  // the best trial's partner slot (bits 0-7) and gluon splitter (bit 8), as screened
  int trials, dipoles;
};

__device__ __forceinline__ void screen_none(Screen& sc) {
  sc.h1 = sc.h2 = INFINITY;
  sc.invc = 0.0f;
  sc.best_code = -1;
  sc.best_hi = sc.best_lo = 0;
  sc.best_aux = 0;
  sc.trials = sc.dipoles = 0;
}

// What the screen reads of one parton: flavour, colour partners and the
// FP32 cache entries of its two dipoles (read whether or not a partner
// exists; the entry is then ignored).
struct PartonScreen {
  int8_t flav;
  uint8_t link0, link1;
  float2 d0, d1;
};

__device__ __forceinline__ PartonScreen load_parton_screen(const Events& E, int64_t ev, int i) {
  PartonScreen q;
  q.flav = E.flav[E.at(i, ev)];
  q.link0 = E.link[E.link_at(0, i, ev)];
  q.link1 = E.link[E.link_at(1, i, ev)];
  q.d0 = E.dip[dip_at(E, 0, i, ev)];
  q.d1 = E.dip[dip_at(E, 1, i, ev)];
  return q;
}

// The loads of the next parton are issued before the trials of the current
// one are generated, so their latency hides behind the Philox rounds.
template <int kMode>
__device__ __forceinline__ void screen_partons(const DevParams& P, const Events& E, int64_t ev, const EventKey& key,
                                               int step, int n, int first, int stride, Screen& sc,
                                               const PartonScreen* first_loaded = nullptr) {
  screen_none(sc);
  if (first >= n) return;
  constexpr float kInvCF2 = static_cast<float>(1.0 / (2.0 * kCF));
  constexpr float kInvCA = static_cast<float>(1.0 / kCA);
  PartonScreen cur = first_loaded ? *first_loaded : load_parton_screen(E, ev, first);
  for (int i = first; i < n; i += stride) {
    PartonScreen nxt = cur;
    if (i + stride < n) nxt = load_parton_screen(E, ev, i + stride);
    const bool gluon = cur.flav == kGluon;
    const bool combined = gluon && per_dipole<kMode>(P);
    const int nk = gluon && !combined ? 1 + P.nf : 1;
    for (int side = 0; side < 2; ++side) {
      if ((side ? cur.link1 : cur.link0) == kNoLink) continue;
      const float2 d = side ? cur.d1 : cur.d0;
      if (d.x < 0.0f) continue;
      ++sc.dipoles;
      // per-dipole trial of a gluon: 1/c of all its kernels (a few ulp)
      const float inv_sum = combined ? 1.0f / (static_cast<float>(kCA) / d.x + static_cast<float>(P.nf) / d.y) : 0.0f;
      for (int kp = 0; kp < nk; kp += 2) {
        const U4 r = philox_draw<kMode>(P, key, static_cast<uint32_t>(step),
                                        static_cast<uint32_t>((2 * i + side) * 4 + kp / 2), kDrawTrial);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int kappa = kp + h;
          if (kappa >= nk) break;
          const uint32_t whi = h ? r.z : r.x, wlo = h ? r.w : r.y;
          const float invc = combined ? inv_sum : (!gluon ? d.x * kInvCF2 : (kappa == 0 ? d.x * kInvCA : d.y));
          const float bound = trial_bound(whi, wlo, invc);
          ++sc.trials;
          const bool first_now = bound < sc.h1;
          sc.h2 = fminf(sc.h2, fmaxf(sc.h1, bound));
          sc.h1 = fminf(sc.h1, bound);
          sc.invc = first_now ? invc : sc.invc;
          sc.best_code = first_now ? (2 * i + side) * 8 + kappa : sc.best_code;
          sc.best_hi = first_now ? whi : sc.best_hi;
          sc.best_lo = first_now ? wlo : sc.best_lo;
          sc.best_aux =
              first_now ? static_cast<uint32_t>(side ? cur.link1 : cur.link0) | (gluon ? 256u : 0u) : sc.best_aux;
        }
      }
    }
    cur = nxt;
  }
}

// Merge the screen of other trials into sc.
__device__ __forceinline__ void screen_merge(Screen& sc, const Screen& o) {
  const bool o_wins = o.h1 < sc.h1;
  sc.h2 = fminf(fminf(sc.h2, o.h2), fmaxf(sc.h1, o.h1));
  if (o_wins) {
    sc.h1 = o.h1;
    sc.invc = o.invc;
    sc.best_code = o.best_code;
    sc.best_hi = o.best_hi;
    sc.best_lo = o.best_lo;
    sc.best_aux = o.best_aux;
  }
  sc.trials += o.trials;
  sc.dipoles += o.dipoles;
}

// Butterfly merge of the screens of the L lanes of each aligned lane group
// (every lane of the warp must call it).
template <int L>
__device__ __forceinline__ void screen_group_reduce(Screen& sc) {
#pragma unroll
  for (int off = 1; off < L; off <<= 1) {
    Screen o;
    o.h1 = __shfl_xor_sync(0xffffffffu, sc.h1, off);
    o.h2 = __shfl_xor_sync(0xffffffffu, sc.h2, off);
    o.invc = __shfl_xor_sync(0xffffffffu, sc.invc, off);
    o.best_code = __shfl_xor_sync(0xffffffffu, sc.best_code, off);
    o.best_hi = __shfl_xor_sync(0xffffffffu, sc.best_hi, off);
    o.best_lo = __shfl_xor_sync(0xffffffffu, sc.best_lo, off);
    o.best_aux = __shfl_xor_sync(0xffffffffu, sc.best_aux, off);
    o.trials = __shfl_xor_sync(0xffffffffu, sc.trials, off);
    o.dipoles = __shfl_xor_sync(0xffffffffu, sc.dipoles, off);
    screen_merge(sc, o);
  }
}

// a > b for numbers (b not -0), from their bits put in order: the FP64 pipe's
// compares cost as much as its FMAs.
__device__ __forceinline__ bool above(double a, double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  return (x ^ ((x >> 63) & 0x7fffffffffffffffll)) > (y ^ ((y >> 63) & 0x7fffffffffffffffll));
}

// What the FP32 screen settles about a cycle: no trial above the cutoff, a
// certain winner (its exact scale computed), or neither -- then the exact
// FP64 selection decides (select_winner_fp64 / fallback_warp).
enum : int { kScreenNone = 0, kScreenWinner = 1, kScreenUndecided = 2 };

// The screen's verdict; for a certain winner its exact scale (from the FP64
// cache) and the winner's data in `task`.  Writes nothing to the record.
// h1, invc: the smallest |key| bound and its trial's 1/c; h2: the smallest
// bound of the other trials; best_code < 0: no trial.
template <int kMode>
__device__ __forceinline__ int screen_verdict(const DevParams& P, const Events& E, int64_t ev, double lnt, float h1,
                                              float h2, float invc, int best_code, uint32_t best_aux, uint32_t best_hi,
                                              uint32_t best_lo, EmitTask& task) {
  // the best trial's key bounds -- |key| - m = h1 and, from it, |key| + m --
  // and the others' upper bound
  const float best_ub = -h1, best_lb = -(fmaf(2.0f * kKeyRelInvc, invc, h1) * (1.0f + 2.1f * kKeyRelKey));
  const float others_hi = -h2;
  // Cutoff threshold in key units: t' > t_C  <=>  key > log2(t_C / t).
  const float lt2 = f32_from_f64(lnt) * 1.44269504f;
  const float thr = P.lg2_tc_f - lt2;
  const float thr_m = 2e-6f * (1.0f + fabsf(lt2) + fabsf(P.lg2_tc_f));

  if (best_code < 0 || fmaxf(best_ub, others_hi) < thr - thr_m) {
    return kScreenNone;  // certainly no trial above the cutoff
  }
  if (best_lb > thr + thr_m && others_hi < best_lb) {
    // Certain winner: its scale exactly, from the FP64 cache.
    const int dcode = best_code >> 3, kappa = best_code & 7;
    const int i = dcode >> 1, side = dcode & 1;
    const int k = static_cast<int>(best_aux & 255u);
    const DipoleRecord rec = E.drec[E.at(side == 0 ? i : k, ev)];
    const bool gluon = (best_aux & 256u) != 0u;  // as the screen read them: no second load
    const bool combined = gluon && per_dipole<kMode>(P);
    const int kind = combined ? kKindUnchosen : (gluon ? (kappa == 0 ? kGtoGG : kGtoQQ) : kQtoQG);
    const double inv_c =
        combined ? inv_c_sum_fp64(P, rec.zp, rec.ls) : inv_c_fp64(P, kind, rec.zp, rec.inv_ls);
    const double lt = fma(log_fp64(to_unit(best_hi, best_lo)), inv_c, lnt);
    if (above(lt, P.ln_tc)) {
      task.lnt = lt;
      task.q2 = rec.q2;
      task.zp = rec.zp;
      task.ls = rec.ls;
      task.i = i;
      task.k = k;
      task.side = side;
      task.kappa = kappa;
      task.kind = kind;
      return kScreenWinner;
    }
  }
  return kScreenUndecided;
}

// What a cycle reads of an event's own state, loaded together: a load behind
// a store to another array is not moved before it, and each would wait for
// its own trip to L2.
struct EventState {
  double lnt;
  unsigned long long hash;
  int trials, dipoles, winners;
};
__device__ __forceinline__ EventState load_state(const Events& E, int64_t ev) {
  return EventState{E.lnt[ev], E.hash[ev], E.n_trials[ev], E.n_dipoles[ev], E.n_winners[ev]};
}

// The first part of the cycle once the screen is known: the cycle and work
// counts, and the screen's verdict.
template <int kMode>
__device__ inline int cycle_screen(const DevParams& P, const Events& E, int64_t ev, int step, const EventState& st,
                                   const Screen& sc, EmitTask& task) {
  E.n_steps[ev] = step + 1;
  E.n_trials[ev] = st.trials + sc.trials;
  E.n_dipoles[ev] = st.dipoles + sc.dipoles;
  const double lnt = st.lnt;
  return screen_verdict<kMode>(P, E, ev, lnt, sc.h1, sc.h2, sc.invc, sc.best_code, sc.best_aux, sc.best_hi, sc.best_lo,
                               task);
}

// The exact FP64 selection for the undecided events of a warp, each computed
// by the whole warp: for every lane whose `need` is set, in turn, lane l takes
// partons l, l + 32, ... of that lane's event and the warp keeps the highest
// scale (the first trial in loop order on ties), the serial selection's
// winner.  The rare undecided cycle of an event with many partons thus takes
// a thirty-second of the dependent loads and FP64 work on its lane, which a
// whole launch or pool would otherwise wait for.  Sets have / task on the
// needing lanes.  Every lane of the warp must call it.
template <int kMode>
__device__ __noinline__ void fallback_warp(const DevParams& P0, const Events& E, bool need, int64_t ev, int job,
                                           EventKey key, int step, int n, double lnt, bool& have, EmitTask& task) {
  const int lane = static_cast<int>(threadIdx.x & 31);
  unsigned pending = __ballot_sync(0xffffffffu, need);
  while (pending) {
    const int src = __ffs(pending) - 1;
    pending &= pending - 1;
    const long long sev = __shfl_sync(0xffffffffu, static_cast<long long>(ev), src);
    EventKey skey;
    skey.id = __shfl_sync(0xffffffffu, key.id, src);
    skey.k0 = kJobKey<kMode> ? __shfl_sync(0xffffffffu, key.k0, src) : 0u;
    skey.k1 = kJobKey<kMode> ? __shfl_sync(0xffffffffu, key.k1, src) : 0u;
    const int sjob = kJobPhysics<kMode> ? __shfl_sync(0xffffffffu, job, src) : 0;
    const int sstep = __shfl_sync(0xffffffffu, step, src);
    const int sn = __shfl_sync(0xffffffffu, n, src);
    const double slnt = __shfl_sync(0xffffffffu, lnt, src);
    const DevParams& P = job_params<kJobPhysics<kMode>>(P0, E, sjob);
    EmitTask w;
    double best = P.ln_tc;
    int code = 0x7fffffff;
    const bool found = select_winner_fp64_range<kMode>(P, E, sev, skey, sstep, sn, slnt, lane, 32, w, best, code);
    // the highest scale; equal scales go to the smallest code
    double wb = best;
    int wc = code;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, wb, off);
      const int oc = __shfl_xor_sync(0xffffffffu, wc, off);
      if (ob > wb || (ob == wb && oc < wc)) {
        wb = ob;
        wc = oc;
      }
    }
    const unsigned own = __ballot_sync(0xffffffffu, found && code == wc);
    if (own) {
      const int ol = __ffs(own) - 1;
      const double t_lnt = __shfl_sync(0xffffffffu, w.lnt, ol), t_q2 = __shfl_sync(0xffffffffu, w.q2, ol);
      const double t_zp = __shfl_sync(0xffffffffu, w.zp, ol);
      const double t_ls = __shfl_sync(0xffffffffu, w.ls, ol);
      const uint32_t packed = __shfl_sync(0xffffffffu,
                                          static_cast<uint32_t>(w.i) | (static_cast<uint32_t>(w.k) << 8) |
                                              (static_cast<uint32_t>(w.side) << 16) |
                                              (static_cast<uint32_t>(w.kappa) << 20) |
                                              (static_cast<uint32_t>(w.kind) << 24),
                                          ol);
      if (lane == src) {
        task.lnt = t_lnt;
        task.q2 = t_q2;
        task.zp = t_zp;
        task.ls = t_ls;
        task.i = static_cast<uint8_t>(packed & 255u);
        task.k = static_cast<uint8_t>((packed >> 8) & 255u);
        task.side = static_cast<uint8_t>((packed >> 16) & 15u);
        task.kappa = static_cast<uint8_t>((packed >> 20) & 15u);
        task.kind = static_cast<uint8_t>(packed >> 24);
      }
    }
    if (lane == src) have = own != 0u;
  }
}

// AcceptOrVeto of a known winner (its data in task): the kernel of a
// per-dipole trial drawn (kind and kappa then written to task), z and the
// acceptance ratio, and the decision added to the event's hash.  Returns
// whether the emission is accepted.  The words of z's
// uniform go to task.  Writes nothing to the record.
template <int kMode>
__device__ __forceinline__ bool accept_or_veto(const DevParams& P, const Events& E, const EventKey& key, int step,
                                               EmitTask& task, unsigned long long& hash) {
  if (task.kind == kKindUnchosen) {
    // per-dipole trial of a gluon: its kernel from the winner's second draw
    const U4 rk = philox_draw<kMode>(P, key, static_cast<uint32_t>(step), 1u, kDrawWinner);
    const int kappa = choose_kernel(P, task.zp, task.ls, to_unit(rk.z, rk.w));
    task.kappa = static_cast<uint8_t>(kappa);
    task.kind = static_cast<uint8_t>(kappa == 0 ? kGtoGG : kGtoQQ);
  }

  // ---- AcceptOrVeto: FP32 screen of Eq. (A.8)-(A.9), FP64 near the edge.
  const U4 rw = philox_draw<kMode>(P, key, static_cast<uint32_t>(step), 0u, kDrawWinner);
  bool accept;
  {
    // z- = t_C / (Q^2 z+) (the same as 1 - z+, without its cancellation);
    // quotients by the two-ulp __fdividef.
    const float zpf = seed_of(task.zp);  // z+ in [1/2, 1]
    const float q2f = f32_from_f64(task.q2);
    const float zmf = __fdividef(P.tcf, q2f * zpf);
    const float rzf = unit_float(rw.x, rw.y);
    float z, e;  // z and 1 - z
    if (task.kind == kGtoQQ) {
      z = fmaf(zpf - zmf, rzf, zmf);
      e = fmaf(-(zpf - zmf), rzf, zpf);
    } else {
      const float x = -rzf * f32_from_f64(task.ls);
      z = fmaf(-zpf, expm1f(x), zmf);
      e = zpf * __expf(x);
    }
    const float lnt_f = f32_from_f64(task.lnt);
    const float y = __fdividef(__expf(lnt_f), q2f * z * e);
    const float as_ratio = P.fixed ? 1.0f : __fdividef(P.as_mz_over_f, fmaf(P.as_b0_f, lnt_f - P.ln_mz2_f, 1.0f));
    float pr;  // P(z, y) / P^over(z)
    if (task.kind == kGtoQQ) {
      pr = fmaf(-2.0f * z, e, 1.0f);
    } else {
      const float soft = __fdividef(e, fmaf(z, y, e));
      pr = task.kind == kQtoQG ? fmaf(-0.5f * (1.0f + z), e, soft) : fmaf(0.5f * z * e, e, soft - e);
    }
    const float ratio = (1.0f - y) * as_ratio * pr;
    const float rvf = unit_float(rw.z, rw.w);
    const float margin = kVetoRel * (fabsf(ratio) + rvf) + kVetoAbs;
    if (fabsf(y - 1.0f) <= 1e-4f || fabsf(rvf - ratio) <= margin) {
      atomicAdd(&E.counters[3], 1ull);  // veto decided in FP64
      accept = accept_fp64(P, task.kind, task.lnt, task.q2, task.zp, task.ls, to_unit(rw.x, rw.y),
                           to_unit(rw.z, rw.w));
    } else {
      accept = y < 1.0f && rvf < ratio;
    }
  }
  hash = fnv1a64(hash, static_cast<uint32_t>(step), task.i, task.side, task.kappa, accept ? 1u : 0u);
  task.rz_hi = rw.x;
  task.rz_lo = rw.y;
  return accept;
}

// The rest of the cycle once the winner is known (have: a trial above t_C,
// with its data in task): CheckCutoff, AcceptOrVeto and the decision hash.
// Returns kCycleFinished when the event left the active state (status
// written), kCycleAccepted with `task` filled when an emission must be
// generated, kCycleVetoed otherwise.
template <int kMode>
__device__ inline int cycle_conclude(const DevParams& P, const Events& E, int64_t ev, const EventKey& key, int step,
                                     int n, const EventState& st, bool have, EmitTask& task) {
  // ---- CheckCutoff.
  if (!have) {
    finish_event(E, ev, GAPS_DONE, P.tc);
    return kCycleFinished;
  }
  E.lnt[ev] = task.lnt;
  E.n_winners[ev] = st.winners + 1;
  unsigned long long hash = st.hash;
  const bool accept = accept_or_veto<kMode>(P, E, key, step, task, hash);
  E.hash[ev] = hash;
  if (!accept) return kCycleVetoed;
  if (n >= E.cap) {
    finish_early(E, ev, GAPS_OVERFLOW, task.lnt);
    return kCycleFinished;
  }
  task.ev = static_cast<int32_t>(ev);
  task.n = n;
  task.step = step;
  return kCycleAccepted;
}

// The whole decision of a cycle in one thread, the exact selection serial.
template <int kMode>
__device__ inline int cycle_decide(const DevParams& P, const Events& E, int64_t ev, const EventKey& key, int step,
                                   int n, const EventState& st, const Screen& sc, EmitTask& task) {
  const int s = cycle_screen<kMode>(P, E, ev, step, st, sc, task);
  bool have = s == kScreenWinner;
  if (s == kScreenUndecided) {
    atomicAdd(&E.counters[2], 1ull);  // screen undecided: full FP64 cycle
    have = select_winner_fp64<kMode>(P, E, ev, key, step, n, st.lnt, task);
  }
  return cycle_conclude<kMode>(P, E, ev, key, step, n, st, have, task);
}

// Phase 1 of a cycle for active event ev, one thread: SelectWinnerEmission
// (the FP32 screen over every trial), then cycle_decide.
template <int kMode>
__device__ inline int cycle_select_veto(const DevParams& P0, const Events& E, int64_t ev, EmitTask& task) {
  const int job = kJobKey<kMode> ? static_cast<int>(E.job_of[ev]) : 0;
  const DevParams& P = job_params<kJobPhysics<kMode>>(P0, E, job);
  const EventKey key = event_key<kMode>(P, E, ev, job);
  const int n = E.n_partons[ev];
  const int step = E.n_steps[ev];
  const EventState st = load_state(E, ev);
  if (step >= P.max_steps) {
    finish_early(E, ev, GAPS_STEP_LIMIT, st.lnt);
    return kCycleFinished;
  }
  Screen sc;
  screen_partons<kMode>(P, E, ev, key, step, n, 0, 1, sc);
  return cycle_decide<kMode>(P, E, ev, key, step, n, st, sc, task);
}

// The splitting variables of an accepted emission: z, y and the azimuth's
// sine and cosine.
struct Splitting {
  double z, y, sphi, cphi;
};
template <int kMode>
__device__ __forceinline__ Splitting splitting_of(const DevParams& P, const EventKey& key, const EmitTask& w) {
  Splitting v;
  const double t = exp_fp64(w.lnt);
  v.z = z_fp64(w.kind, w.zp, w.ls, to_unit(w.rz_hi, w.rz_lo));
  v.y = div_fp64(t, w.q2 * v.z * (1.0 - v.z));
  const U4 rphi = philox_draw<kMode>(P, key, static_cast<uint32_t>(w.step), 1u, kDrawWinner);
  circle_fp64(to_unit(rphi.x, rphi.y), rphi.x, &v.sphi, &v.cphi);
  return v;
}

// What emit_colours reads of the record: the partners of the splitter and of
// the spectator outside their dipole (the colour chain is open, so i, j, k
// and these are distinct), the splitter's colour line on j's side, the next
// free line and the emissions so far.  Loaded together, ahead of the FP64
// work, as EventState is.
struct EmitState {
  int oi, ok, line, colour, emissions;
};
__device__ __forceinline__ EmitState load_emit_state(const Events& E, const EmitTask& w) {
  const int64_t ev = w.ev;
  const int s = w.kind == kGtoQQ ? 1 : w.side;
  return EmitState{E.link[E.link_at(1 - w.side, w.i, ev)], E.link[E.link_at(w.side, w.k, ev)],
                   (s ? E.acol : E.col)[E.at(w.i, ev)], E.next_colour[ev], E.n_emissions[ev]};
}

// Colours, links and flavours of an emission, its refresh list and counts.
//
// A gluon enters the shared colour line between splitter and spectator: on
// side `s` it takes the splitter's line and on the other a new line m, the
// splitter takes m on side s.  g(c, a) -> q(c, 0) + qbar(0, a) is the same on
// the anticolour side with no line m: the antiquark connects to the holder of
// colour a, and not to the quark.
template <class Reserve, class Put>
__device__ __forceinline__ void emit_colours(const Events& E, const EmitTask& w, const EmitState& st,
                                             Reserve reserve, Put put, int task_index) {
  const int64_t ev = w.ev;
  const int i = w.i, j = w.n, k = w.k, side = w.side;
  const bool split = w.kind == kGtoQQ;
  const int s = split ? 1 : side;
  const int oi = st.oi, ok = st.ok;
  const int to = split && side == 0 ? oi : k;  // j's partner on side s
  const int m = split ? 0 : st.colour;
  if (!split) E.next_colour[ev] = m + 1;
  const size_t ai = E.at(i, ev), aj = E.at(j, ev);
  int16_t* line = s ? E.acol : E.col;
  int16_t* other = s ? E.col : E.acol;
  line[aj] = static_cast<int16_t>(st.line);
  other[aj] = static_cast<int16_t>(m);
  line[ai] = static_cast<int16_t>(m);
  E.link[E.link_at(s, i, ev)] = split ? kNoLink : static_cast<uint8_t>(j);
  E.link[E.link_at(s, j, ev)] = static_cast<uint8_t>(to);
  E.link[E.link_at(1 - s, j, ev)] = split ? kNoLink : static_cast<uint8_t>(i);
  E.link[E.link_at(1 - s, to, ev)] = static_cast<uint8_t>(j);
  if (split) E.flav[ai] = static_cast<int8_t>(w.kappa);
  E.flav[aj] = static_cast<int8_t>(split ? -w.kappa : kGluon);
  // Every dipole with a moved parton, once.  A gluon: (i, j), (j, k) and the
  // outer ones of i and k.  A splitting: the quark's on its colour side, the
  // antiquark's on its anticolour side -- one of them to the spectator, the
  // other the gluon's outer one -- and the spectator's outer one.
  int at = reserve(2 + (!split && oi != kNoLink ? 1 : 0) + (ok != kNoLink ? 1 : 0));
  put(at++, split ? pack_refresh(task_index, i, 0, side == 0 ? k : oi) : pack_refresh(task_index, i, side, j));
  put(at++, pack_refresh(task_index, j, s, to));
  if (!split && oi != kNoLink) put(at++, pack_refresh(task_index, i, 1 - side, oi));
  if (ok != kNoLink) put(at++, pack_refresh(task_index, k, side, ok));
  E.n_partons[ev] = j + 1;
  E.n_emissions[ev] = st.emissions + 1;
}

// Phase 2: GenerateEmission -- azimuth, the final-final dipole map, colours
// and the new parton in slot n.  The dipoles whose invariant mass moved are
// put in the block's refresh list (reserve(count) gives their first place,
// put(place, job) writes one) under task_index; the caller recomputes them
// after a block barrier, spread over all of its threads, so that this
// FP64-heavy step runs in full warps.
template <int kMode, class Reserve, class Put>
__device__ inline void cycle_emit(const DevParams& P0, const Events& E, const EmitTask& w, Reserve reserve, Put put,
                                  int task_index) {
  const int64_t ev = w.ev;
  const int job = kJobKey<kMode> ? static_cast<int>(E.job_of[ev]) : 0;
  const DevParams& P = job_params<kJobPhysics<kMode>>(P0, E, job);
  const Splitting v = splitting_of<kMode>(P, event_key<kMode>(P, E, ev, job), w);
  const int i = w.i, j = w.n, k = w.k;
  const V4 a = load_p(E, i, ev);
  const V4 b = load_p(E, k, ev);
  const EmitState st = load_emit_state(E, w);
  V4 pi, pj, pb;
  dipole_map(a, b, v.z, v.y, v.cphi, v.sphi, pi, pj, pb);
  store_p(E, i, ev, pi);
  store_p(E, j, ev, pj);
  store_p(E, k, ev, pb);
  emit_colours(E, w, st, reserve, put, task_index);
}

// GenerateEmission by four lanes a task, lane c of a group with momentum
// component c, for lists too short to fill warps with a task per thread.  A
// warp issues an FP64 instruction every 64 cycles whatever its active lanes,
// so a short list waits for the number of them on its chain: 161 for a task
// in one lane.  Four lanes take about 90, and about 60 where one warp forms
// the frame and the momenta and another the splitting variables and the
// colours.  Each value comes from the operations of cycle_emit in their
// order, so the events are the same.  Every lane of a warp calls these, the
// lanes of groups without a task with another's and has = false.
//
// The splitting variables, on every lane of the group: splitting_of with the
// two exponentials on two lanes, and kt = sqrt(z (1 - z) y Q^2) of
// dipole_map.  trig: cosine, sine of the azimuth.
struct Splitting4 {
  double z, y, kt, trig[2];
};
template <int kMode>
__device__ __forceinline__ Splitting4 splitting_of4(const DevParams& P, const EventKey& key, const EmitTask& w,
                                                    const V4& a, const V4& b, int c) {
  Splitting4 v;
  const double r = to_unit(w.rz_hi, w.rz_lo);
  const double ex = exp_or_expm1_fp64(c == 0 ? w.lnt : -r * w.ls, c != 0);
  const double t = __shfl_sync(0xffffffffu, ex, 0, 4), em = __shfl_sync(0xffffffffu, ex, 1, 4);
  const double zm = 1.0 - w.zp;
  const bool split = w.kind == kGtoQQ;  // as z_fp64
  v.z = fma(split ? w.zp - zm : -w.zp, split ? r : em, zm);
  v.y = div_fp64(t, w.q2 * v.z * (1.0 - v.z));
  const U4 rphi = philox_draw<kMode>(P, key, static_cast<uint32_t>(w.step), 1u, kDrawWinner);
  circle_fp64(to_unit(rphi.x, rphi.y), rphi.x, &v.trig[1], &v.trig[0]);
  v.kt = sqrt_fp64(v.z * (1.0 - v.z) * v.y * (2.0 * mdot(a, b)));
  return v;
}

// The momenta from the frame (dipole_frame4) and the splitting variables.
__device__ __forceinline__ void emit_momenta4(const Events& E, const EmitTask& w, const V4& a, const V4& b, int c,
                                              double n1c, double n2c, double inv, const Splitting4& v, bool has) {
  const double kk = v.kt * v.trig[c >> 1] * inv;
  const double kc = __shfl_sync(0xffffffffu, kk, 0, 4), ks = __shfl_sync(0xffffffffu, kk, 2, 4);
  const double q = fma(ks, n2c, kc * n1c);
  const double ac = component(a, c), bc = component(b, c);
  const double fa_j = 1.0 - v.z, fb_i = fa_j * v.y, fb_j = v.z * v.y;
  double* out = c == 0 ? E.e : (c == 1 ? E.px : (c == 2 ? E.py : E.pz));
  if (!has) return;
  out[E.at(w.i, w.ev)] = fma(fb_i, bc, fma(v.z, ac, q));
  out[E.at(w.n, w.ev)] = fma(fb_j, bc, fma(fa_j, ac, -q));
  out[E.at(w.k, w.ev)] = (1.0 - v.y) * bc;
}

// One warp, up to 8 tasks: w is the task of the calling lane's group.
template <int kMode, class Reserve, class Put>
__device__ inline void emit_warp4(const DevParams& P0, const Events& E, const EmitTask& w, bool has, Reserve reserve,
                                  Put put, int task_index) {
  const int c = static_cast<int>(threadIdx.x & 3);
  const int64_t ev = w.ev;
  const int job = kJobKey<kMode> ? static_cast<int>(E.job_of[ev]) : 0;
  const DevParams& P = job_params<kJobPhysics<kMode>>(P0, E, job);
  const V4 a = load_p(E, w.i, ev);
  const V4 b = load_p(E, w.k, ev);
  const EmitState st = load_emit_state(E, w);
  double n1c, n2c, inv;
  dipole_frame4(a, b, c, n1c, n2c, inv);
  const Splitting4 v = splitting_of4<kMode>(P, event_key<kMode>(P, E, ev, job), w, a, b, c);
  emit_momenta4(E, w, a, b, c, n1c, n2c, inv, v, has);
  if (has && c == 0) emit_colours(E, w, st, reserve, put, task_index);
}

// Two warps (the first 64 threads of a block, with `sync` a barrier), up to 8
// tasks: tasks[0 .. count), count > 0; splits: shared memory.  Plain shower
// 10^3 events 1.03 -> 0.87 ms against a task per lane, 1.2x10^4 (200 GeV)
// 3.65 -> 3.38, 10^5 2.63 -> 2.47; taken for lists of up to 16 tasks a block
// it measured the same, up to 32 it slows 10^5 events to 2.70 ms.
template <int kMode, class Reserve, class Put, class Sync>
__device__ inline void emit_shared(const DevParams& P0, const Events& E, const EmitTask* tasks, int count,
                                   Splitting4* splits, int tid, Reserve reserve, Put put, Sync sync) {
  const int g = (tid & 31) >> 2, c = tid & 3, index = min(g, count - 1);
  const bool has = g < count;
  const EmitTask& w = tasks[index];
  const int64_t ev = w.ev;
  const V4 a = load_p(E, w.i, ev);
  const V4 b = load_p(E, w.k, ev);
  // the frame's warp and the splitting variables' meet at one barrier that
  // the whole block passes, not at one in each branch
  const bool frame = tid < 32;
  double n1c = 0.0, n2c = 0.0, inv = 0.0;
  EmitState st{};
  if (frame) {
    dipole_frame4(a, b, c, n1c, n2c, inv);
  } else {
    const int job = kJobKey<kMode> ? static_cast<int>(E.job_of[ev]) : 0;
    const DevParams& P = job_params<kJobPhysics<kMode>>(P0, E, job);
    st = load_emit_state(E, w);
    const Splitting4 v = splitting_of4<kMode>(P, event_key<kMode>(P, E, ev, job), w, a, b, c);
    if (has && c == 0) splits[g] = v;
  }
  sync();
  if (frame) {
    emit_momenta4(E, w, a, b, c, n1c, n2c, inv, splits[index], has);
  } else if (has && c == 0) {
    emit_colours(E, w, st, reserve, put, g);
  }
}

// One dipole of the refresh list.
// refresh_task: the position, in the caller's queue, of the task whose event
// the job belongs to.
__device__ __forceinline__ int refresh_task(uint32_t job) { return static_cast<int>(job & 1023u); }
// The invariant mass of a refresh job's dipole from the stored momenta of its
// two partons (the oracle's formula, in the oracle's operand order).
__device__ __forceinline__ double refresh_mass(const Events& E, int64_t ev, uint32_t job) {
  const int x = static_cast<int>((job >> 10) & 255u), k = static_cast<int>((job >> 18) & 255u);
  return 2.0 * mdot(load_p(E, x, ev), load_p(E, k, ev));
}
__device__ __forceinline__ void refresh_store(const Events& E, int64_t ev, uint32_t job, const DipoleEntry& d) {
  const int x = static_cast<int>((job >> 10) & 255u);
  const int k = static_cast<int>((job >> 18) & 255u), side = static_cast<int>((job >> 26) & 1u);
  store_dipole(E, ev, x, side, k, d);
}
template <bool kMulti>
__device__ inline void refresh_dipole(const DevParams& P0, const Events& E, int64_t ev, uint32_t job) {
  const DevParams& P = params_of<kMulti>(P0, E, ev);
  refresh_store(E, ev, job, make_dipole(P, refresh_mass(E, ev, job)));
}

}  // namespace gaps

// Observables of the finished events (Sec. 3.1): exact thrust and the
// heavy-jet mass, and the Durham jet resolutions y23..y56.
//
// Layout of the work.  The finished events are first bucketed by parton
// multiplicity (count, scan, scatter into an index list), so the threads of
// a warp handle events of the same size: the O(n^3) loops of thrust and
// Durham then run with no lane waiting on a larger neighbour.  Events of up
// to 16 partons take one thread each, with per-thread arrays (in batches of
// fewer than 180 000 events, groups of 4 to 16 lanes: the event's momenta sit in
// shared memory, the lanes split the pairs of each search and reduce their
// partial results in the serial loop's order, and the O(n) FP64 sums run one
// component per lane in that order, so the results are the one-thread
// results).  Larger events take a warp each (event_shapes_warp), with the O(n)
// steps spread over the lanes and a nearest-neighbour table in the clustering.
//
// Precision.  As in the shower, the searches run in FP32 and the answers in
// FP64:
//  * Thrust.  Every candidate partition P = sum s_i p_i of the exact
//    algorithm (planes through every pair, both signs of the pair) is scored
//    |P|^2 in FP32 and identified by its bitmask; the best distinct
//    partitions are tracked.  When the best beats the runner-up by more than
//    the FP32 error bound (or, in large events, is the longest of those within
//    it), its |P| and axis are recomputed in FP64; otherwise the whole search
//    runs in FP64.
//    A momentum within FP32 rounding of a pair's plane may get the wrong side,
//    which that bound does not cover: above 16 partons the sides in doubt are
//    decided in FP64, pair by pair (sides_fp32, sides_fp64), so that the search
//    sees the exact algorithm's partitions; the winner must also be the
//    partition that its own axis defines.  Up to 16 partons every partition
//    has to be missed by all its pairs to go unseen: sides are as FP32 has them.
//  * Durham.  Pair distances min(E_i^2, E_j^2) |u_i - u_j|^2 (u = unit
//    momentum, free of the 1 - cos cancellation) are compared in FP32 with a
//    per-pair error bound; every pair that could be the minimum is evaluated
//    with the FP64 formula 2 min(E_i^2, E_j^2)(1 - cos theta_ij)/s, and the
//    smallest of those is merged, ties to the first pair as in the oracle.
//  * Final scalings take reciprocals (1/s, 1/|P|, 1/(2 sum |p|)): the
//    oracle's divisions up to an ulp.  The cosine inside Durham's 1 - cos
//    keeps the oracle's division, since 1 - cos magnifies its rounding.
#include <type_traits>

#include "gaps_launch.hpp"
#include "sqrt_obs.cuh"

namespace gaps {

namespace {

constexpr int kShapeThreads = 128;

// The products and sums of this file in fused form (the library is built
// without automatic contraction): both the per-thread and the lane-group
// forms below call these, so they round alike.
__device__ __forceinline__ float dot3f(float ax, float ay, float az, float bx, float by, float bz) {
  return fmaf(az, bz, fmaf(ay, by, ax * bx));
}
__device__ __forceinline__ float crossf(float a, float b, float c, float d) { return fmaf(a, b, -(c * d)); }
__device__ __forceinline__ double dot3(double ax, double ay, double az, double bx, double by, double bz) {
  return fma(az, bz, fma(ay, by, ax * bx));
}
__device__ __forceinline__ double cross(double a, double b, double c, double d) { return fma(a, b, -(c * d)); }
// The squared mass of a four-vector (e, x, y, z).
__device__ __forceinline__ double mass2(const double* h) {
  return fma(-h[3], h[3], fma(-h[2], h[2], fma(-h[1], h[1], h[0] * h[0])));
}

// Exact FP64 thrust search (the fallback): planes through every pair with a
// non-zero cross product, other momenta signed by their side, the pair tried
// with both signs; the longest P is the thrust axis.
template <int MAXJ>
__device__ double thrust_fp64(int n, const double* jx, const double* jy, const double* jz, double sum_abs,
                              double& ax, double& ay, double& az) {
  double best2 = -1.0, bx = 0.0, by = 0.0, bz = 0.0;
  for (int j = 0; j < n; ++j) {
    for (int k = j + 1; k < n; ++k) {
      const double nx = cross(jy[j], jz[k], jz[j], jy[k]);
      const double ny = cross(jz[j], jx[k], jx[j], jz[k]);
      const double nz = cross(jx[j], jy[k], jy[j], jx[k]);
      if (nx == 0.0 && ny == 0.0 && nz == 0.0) continue;
      double px = 0.0, py = 0.0, pz = 0.0;
      for (int i = 0; i < n; ++i) {
        if (i == j || i == k) continue;
        const double sg = dot3(jx[i], jy[i], jz[i], nx, ny, nz) >= 0.0 ? 1.0 : -1.0;
        px = fma(sg, jx[i], px);
        py = fma(sg, jy[i], py);
        pz = fma(sg, jz[i], pz);
      }
      for (int c = 0; c < 4; ++c) {
        const double fj = (c & 2) ? -1.0 : 1.0, fk = (c & 1) ? -1.0 : 1.0;
        const double cx = fma(fk, jx[k], fma(fj, jx[j], px));
        const double cy = fma(fk, jy[k], fma(fj, jy[j], py));
        const double cz = fma(fk, jz[k], fma(fj, jz[j], pz));
        const double c2 = dot3(cx, cy, cz, cx, cy, cz);
        if (c2 > best2) {
          best2 = c2;
          bx = cx;
          by = cy;
          bz = cz;
        }
      }
    }
  }
  if (best2 < 0.0) {  // collinear: T = 1 along the first momentum
    const double l = sqrt_obs(dot3(jx[0], jy[0], jz[0], jx[0], jy[0], jz[0]));
    ax = jx[0] / l;
    ay = jy[0] / l;
    az = jz[0] / l;
    return 1.0;
  }
  const double l = sqrt_obs(best2), inv_l = 1.0 / l;
  ax = bx * inv_l;
  ay = by * inv_l;
  az = bz * inv_l;
  return l / sum_abs;
}

// Top two distinct partitions by score.
struct Top2 {
  float s1 = -1.0f, s2 = -1.0f;
  unsigned long long m1 = 0ull, m2 = ~0ull;
  __device__ __forceinline__ void add(float s, unsigned long long m) {
    if (m == m1) {
      s1 = fmaxf(s1, s);
    } else if (s > s1) {
      s2 = s1;
      m2 = m1;
      s1 = s;
      m1 = m;
    } else if (m == m2) {
      s2 = fmaxf(s2, s);
    } else if (s > s2) {
      s2 = s;
      m2 = m;
    }
  }
};

template <int MAXJ>
__device__ void event_shapes(const DevParams& P0, const Events& E, int64_t ev, int n) {
  const DevParams& P = params_of_event(P0, E, ev);
  double je[MAXJ], jx[MAXJ], jy[MAXJ], jz[MAXJ], ja[MAXJ];  // ja: |p| of every jet
  float fx[MAXJ], fy[MAXJ], fz[MAXJ];
  double sum_abs = 0.0;
  float sum_absf = 0.0f;
  for (int i = 0; i < n; ++i) {
    const size_t a = E.at(i, ev);
    je[i] = E.e[a];
    jx[i] = E.px[a];
    jy[i] = E.py[a];
    jz[i] = E.pz[a];
    fx[i] = f32_from_f64(jx[i]);
    fy[i] = f32_from_f64(jy[i]);
    fz[i] = f32_from_f64(jz[i]);
    ja[i] = sqrt_obs(dot3(jx[i], jy[i], jz[i], jx[i], jy[i], jz[i]));
    sum_abs += ja[i];
  }
  sum_absf = f32_from_f64(sum_abs);

  // ---- thrust
  double thrust = 1.0, ax = 0.0, ay = 0.0, az = 0.0;
  bool decided = false;
  if (n == 2) {
    // no emission: the pair is back to back, T = 1 along the quark
    const double inv_l = 1.0 / ja[0];
    ax = jx[0] * inv_l;
    ay = jy[0] * inv_l;
    az = jz[0] * inv_l;
    decided = true;
  } else {
    static_assert(MAXJ < 64, "a partition is a word");
    Top2 top;
    const unsigned long long full = (1ull << n) - 1ull;
    for (int j = 0; j < n; ++j) {
      for (int k = j + 1; k < n; ++k) {
        const float nx = crossf(fy[j], fz[k], fz[j], fy[k]);
        const float ny = crossf(fz[j], fx[k], fx[j], fz[k]);
        const float nz = crossf(fx[j], fy[k], fy[j], fx[k]);
        if (nx == 0.0f && ny == 0.0f && nz == 0.0f) continue;
        float px = 0.0f, py = 0.0f, pz = 0.0f;
        unsigned long long mask = 0ull;
        for (int i = 0; i < n; ++i) {
          if (i == j || i == k) continue;
          if (dot3f(fx[i], fy[i], fz[i], nx, ny, nz) >= 0.0f) {
            px += fx[i];
            py += fy[i];
            pz += fz[i];
            mask |= 1ull << i;
          } else {
            px -= fx[i];
            py -= fy[i];
            pz -= fz[i];
          }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const bool pj = !(c & 2), pk = !(c & 1);
          const float cx = px + (pj ? fx[j] : -fx[j]) + (pk ? fx[k] : -fx[k]);
          const float cy = py + (pj ? fy[j] : -fy[j]) + (pk ? fy[k] : -fy[k]);
          const float cz = pz + (pj ? fz[j] : -fz[j]) + (pk ? fz[k] : -fz[k]);
          unsigned long long m = mask | (pj ? 1ull << j : 0ull) | (pk ? 1ull << k : 0ull);
          if (m & 1ull) m = ~m & full;  // a partition and its complement are one candidate
          top.add(dot3f(cx, cy, cz, cx, cy, cz), m);
        }
      }
    }
    // FP32 error of |P|^2: n rounded terms of size <= sum |p| per component.
    const float margin = 8.0f * static_cast<float>(n + 2) * 6.0e-8f * sum_absf * sum_absf;
    if (top.s1 < 0.0f) {
      decided = false;  // no pair spans a plane: let the exact search decide
    } else if (top.s2 < top.s1 - margin) {
      double px = 0.0, py = 0.0, pz = 0.0;
      for (int i = 0; i < n; ++i) {
        const double sg = ((top.m1 >> i) & 1ull) ? 1.0 : -1.0;
        px = fma(sg, jx[i], px);
        py = fma(sg, jy[i], py);
        pz = fma(sg, jz[i], pz);
      }
      const double l = sqrt_obs(dot3(px, py, pz, px, py, pz)), inv_l = 1.0 / l;
      thrust = l / sum_abs;
      ax = px * inv_l;
      ay = py * inv_l;
      az = pz * inv_l;
      decided = true;
    }
  }
  if (!decided) {
    atomicAdd(&E.counters[4], 1ull);  // thrust decided by the exact FP64 search
    thrust = thrust_fp64<MAXJ>(n, jx, jy, jz, sum_abs, ax, ay, az);
  }
  // Hemispheres by the sign of p . n_T: heavy-jet mass, and the jet
  // broadenings B_+- = sum |p x n_T| / (2 sum |p|), B_T = B_+ + B_-,
  // B_W = max(B_+, B_-).
  double hp[4] = {0, 0, 0, 0}, hm[4] = {0, 0, 0, 0};
  double bp = 0.0, bm = 0.0;
  for (int i = 0; i < n; ++i) {
    // p . n >= 0 on the bits (-0 counts as 0; the FP64 pipe's compares cost
    // as much as its FMAs on this part)
    const long long pn = __double_as_longlong(dot3(jx[i], jy[i], jz[i], ax, ay, az));
    const bool plus = pn >= 0 || pn == static_cast<long long>(0x8000000000000000ull);
    double* h = plus ? hp : hm;
    h[0] += je[i];
    h[1] += jx[i];
    h[2] += jy[i];
    h[3] += jz[i];
    const double cx = cross(jy[i], az, jz[i], ay), cy = cross(jz[i], ax, jx[i], az), cz = cross(jx[i], ay, jy[i], ax);
    const double pt = sqrt_obs(dot3(cx, cy, cz, cx, cy, cz));
    if (plus) {
      bp += pt;
    } else {
      bm += pt;
    }
  }
  const double mp = mass2(hp);
  const double mm = mass2(hm);
  E.obs[4 * E.stride + ev] = 1.0 - thrust;
  E.obs[5 * E.stride + ev] = fmax(mp, mm) * P.inv_s;
  const double inv_2sum = 0.5 / sum_abs;
  bp *= inv_2sum;
  bm *= inv_2sum;
  E.obs[6 * E.stride + ev] = bp + bm;
  E.obs[7 * E.stride + ev] = fmax(bp, bm);

  // ---- Durham (E-scheme)
  float fe2[MAXJ];
  for (int i = 0; i < n; ++i) {
    const float e = f32_from_f64(je[i]);
    fe2[i] = e * e;
    const float r = rsqrtf(dot3f(fx[i], fy[i], fz[i], fx[i], fy[i], fz[i]));
    fx[i] *= r;  // from here on fx, fy, fz hold unit directions
    fy[i] *= r;
    fz[i] *= r;
  }
  double yres[4] = {-1.0, -1.0, -1.0, -1.0};
  // y of jets i, j with the oracle's FP64 formula (|p| cached per jet).
  auto y_exact = [&](int i, int j) {
    const double cosij = dot3(jx[i], jy[i], jz[i], jx[j], jy[j], jz[j]) / (ja[i] * ja[j]);
    return 2.0 * fmin(je[i] * je[i], je[j] * je[j]) * (1.0 - cosij) * P.inv_s;
  };
  for (int m = n; m > 2; --m) {  // y of the last two jets is not recorded
    // pass 1: the smallest upper bound of the FP32 distances, and its pair
    float ubest = INFINITY;
    int ui = 0, uj = 1;
    for (int i = 0; i < m; ++i) {
      for (int j = i + 1; j < m; ++j) {
        const float dx = fx[i] - fx[j], dy = fy[i] - fy[j], dz = fz[i] - fz[j];
        const float d = dot3f(dx, dy, dz, dx, dy, dz);
        const float y = fminf(fe2[i], fe2[j]) * d;
        const float rel = 4.0e-6f + 1.0e-6f * rsqrtf(fmaxf(d, 1e-30f));
        const float ub = fmaf(y, 1.0f + rel, 1e-30f);
        if (ub < ubest) {
          ubest = ub;
          ui = i;
          uj = j;
        }
      }
    }
    // pass 2: how many pairs have a lower bound that reaches it
    int n_cand = 0;
    for (int i = 0; i < m; ++i) {
      for (int j = i + 1; j < m; ++j) {
        const float dx = fx[i] - fx[j], dy = fy[i] - fy[j], dz = fz[i] - fz[j];
        const float d = dot3f(dx, dy, dz, dx, dy, dz);
        const float y = fminf(fe2[i], fe2[j]) * d;
        const float rel = 4.0e-6f + 1.0e-6f * rsqrtf(fmaxf(d, 1e-30f));
        n_cand += y * (1.0f - rel) <= ubest ? 1 : 0;
      }
    }
    // One candidate (nearly every merge): it is the pair of the smallest
    // upper bound and the exact minimum, evaluated once, in step with the
    // other lanes.  Otherwise every candidate in FP64, ties to the first
    // pair as in the oracle.
    double ymin = 0.0;
    int bi = ui, bj = uj;
    if (n_cand == 1) {
      if (m <= 6) ymin = y_exact(ui, uj);  // the merges that are recorded
    } else {
      atomicAdd(&E.counters[5], 1ull);  // merges with several FP64 candidates
      bi = -1;
      for (int i = 0; i < m; ++i) {
        for (int j = i + 1; j < m; ++j) {
          const float dx = fx[i] - fx[j], dy = fy[i] - fy[j], dz = fz[i] - fz[j];
          const float d = dot3f(dx, dy, dz, dx, dy, dz);
          const float y = fminf(fe2[i], fe2[j]) * d;
          const float rel = 4.0e-6f + 1.0e-6f * rsqrtf(fmaxf(d, 1e-30f));
          if (y * (1.0f - rel) > ubest) continue;
          const double yy = y_exact(i, j);
          if (bi < 0 || yy < ymin) {
            ymin = yy;
            bi = i;
            bj = j;
          }
        }
      }
    }
    if (m <= 6) yres[m - 3] = ymin;
    if (m == 3) break;
    je[bi] += je[bj];
    jx[bi] += jx[bj];
    jy[bi] += jy[bj];
    jz[bi] += jz[bj];
    je[bj] = je[m - 1];
    jx[bj] = jx[m - 1];
    jy[bj] = jy[m - 1];
    jz[bj] = jz[m - 1];
    ja[bj] = ja[m - 1];
    ja[bi] = sqrt_obs(dot3(jx[bi], jy[bi], jz[bi], jx[bi], jy[bi], jz[bi]));
    fe2[bj] = fe2[m - 1];
    fx[bj] = fx[m - 1];
    fy[bj] = fy[m - 1];
    fz[bj] = fz[m - 1];
    {
      const float e = f32_from_f64(je[bi]);
      fe2[bi] = e * e;
      const float x = f32_from_f64(jx[bi]), y = f32_from_f64(jy[bi]), z = f32_from_f64(jz[bi]);
      const float r = rsqrtf(dot3f(x, y, z, x, y, z));
      fx[bi] = x * r;
      fy[bi] = y * r;
      fz[bi] = z * r;
    }
  }
  for (int h = 0; h < 4; ++h) E.obs[h * E.stride + ev] = yres[h];
}

// ------------------------------------------------------- lane groups
// Lanes of this thread's aligned group of L (L a power of two, < 32).
template <int L>
__device__ __forceinline__ unsigned group_lanes() {
  return ((1u << L) - 1u) << ((threadIdx.x & 31u) & ~static_cast<unsigned>(L - 1));
}

// The pairs (j, k), j < k < n, of one lane: positions sub, sub + L, ... of
// the serial loop (j outer, k inner); p is the position.
struct PairWalk {
  int j, off, row, p;
  __device__ __forceinline__ void start(int n, int sub) {
    j = 0;
    off = sub;
    row = n - 1;
    p = sub;
    settle(n);
  }
  __device__ __forceinline__ void settle(int n) {
    while (j < n - 1 && off >= row) {
      off -= row;
      ++j;
      row = n - 1 - j;
    }
  }
  __device__ __forceinline__ bool valid(int n) const { return j < n - 1; }
  __device__ __forceinline__ int k() const { return j + 1 + off; }
  template <int L>
  __device__ __forceinline__ void next(int n) {
    off += L;
    p += L;
    settle(n);
  }
};

// The event's arrays in shared memory, one set per group.  j: E, px, py, pz;
// ja: |p|; pt, plus: |p x n_T| and the hemisphere of every parton; sums: the
// hemispheres' sums of E, px, py, pz and pt.
template <int MAXJ>
struct GroupArrays {
  double j[4][MAXJ], ja[MAXJ], pt[MAXJ], sums[2][5];
  float fx[MAXJ], fy[MAXJ], fz[MAXJ], fe2[MAXJ];
  uint8_t plus[MAXJ];
};

// thrust_fp64 over the group: each lane takes its pairs, the group keeps the
// longest P and, on equal lengths, the first candidate in the serial loop's
// order (pair position x 4 + sign choice), so the result is the serial one.
template <int MAXJ, int L>
__device__ double thrust_fp64_group(int n, const GroupArrays<MAXJ>& a, double sum_abs, int sub, unsigned gm,
                                    double& ax, double& ay, double& az) {
  double best2 = -1.0, bx = 0.0, by = 0.0, bz = 0.0;
  int bidx = 0x7fffffff;
  PairWalk w;
  for (w.start(n, sub); w.valid(n); w.next<L>(n)) {
    const int j = w.j, k = w.k();
    const double nx = cross(a.j[2][j], a.j[3][k], a.j[3][j], a.j[2][k]);
    const double ny = cross(a.j[3][j], a.j[1][k], a.j[1][j], a.j[3][k]);
    const double nz = cross(a.j[1][j], a.j[2][k], a.j[2][j], a.j[1][k]);
    if (nx == 0.0 && ny == 0.0 && nz == 0.0) continue;
    double px = 0.0, py = 0.0, pz = 0.0;
    for (int i = 0; i < n; ++i) {
      if (i == j || i == k) continue;
      const double sg = dot3(a.j[1][i], a.j[2][i], a.j[3][i], nx, ny, nz) >= 0.0 ? 1.0 : -1.0;
      px = fma(sg, a.j[1][i], px);
      py = fma(sg, a.j[2][i], py);
      pz = fma(sg, a.j[3][i], pz);
    }
    for (int c = 0; c < 4; ++c) {
      const double fj = (c & 2) ? -1.0 : 1.0, fk = (c & 1) ? -1.0 : 1.0;
      const double cx = fma(fk, a.j[1][k], fma(fj, a.j[1][j], px));
      const double cy = fma(fk, a.j[2][k], fma(fj, a.j[2][j], py));
      const double cz = fma(fk, a.j[3][k], fma(fj, a.j[3][j], pz));
      const double c2 = dot3(cx, cy, cz, cx, cy, cz);
      if (c2 > best2) {  // within a lane the positions rise: the first wins ties
        best2 = c2;
        bidx = 4 * w.p + c;
        bx = cx;
        by = cy;
        bz = cz;
      }
    }
  }
#pragma unroll
  for (int off = 1; off < L; off <<= 1) {
    const double o2 = __shfl_xor_sync(gm, best2, off);
    const int oi = __shfl_xor_sync(gm, bidx, off);
    const double ox = __shfl_xor_sync(gm, bx, off), oy = __shfl_xor_sync(gm, by, off);
    const double oz = __shfl_xor_sync(gm, bz, off);
    if (o2 > best2 || (o2 == best2 && oi < bidx)) {
      best2 = o2;
      bidx = oi;
      bx = ox;
      by = oy;
      bz = oz;
    }
  }
  if (best2 < 0.0) {  // collinear: T = 1 along the first momentum
    const double l = sqrt_obs(dot3(a.j[1][0], a.j[2][0], a.j[3][0], a.j[1][0], a.j[2][0], a.j[3][0]));
    ax = a.j[1][0] / l;
    ay = a.j[2][0] / l;
    az = a.j[3][0] / l;
    return 1.0;
  }
  const double l = sqrt_obs(best2), inv_l = 1.0 / l;
  ax = bx * inv_l;
  ay = by * inv_l;
  az = bz * inv_l;
  return l / sum_abs;
}

// event_shapes for one event by a group of L >= 4 lanes (every lane of the
// group calls it for the same event).  The searches give exactly the serial
// results: each lane screens its pairs in the serial order, the group merges
// the lanes' bests with the serial tie rule, and the sums (thrust,
// hemispheres, broadenings, the merged jets) run one component per lane in
// the serial order: a warp can issue an FP64 instruction every 64 cycles
// only, so a lone event's time is their number.  Lane 0 of the group writes
// the observables.
template <int MAXJ, int L>
__device__ void event_shapes_group(const DevParams& P0, const Events& E, int64_t ev, int n, GroupArrays<MAXJ>& a,
                                   int sub, unsigned gm) {
  const DevParams& P = params_of_event(P0, E, ev);
  for (int i = sub; i < n; i += L) {
    const size_t at = E.at(i, ev);
    const double x = E.px[at], y = E.py[at], z = E.pz[at];
    a.j[0][i] = E.e[at];
    a.j[1][i] = x;
    a.j[2][i] = y;
    a.j[3][i] = z;
    a.fx[i] = f32_from_f64(x);
    a.fy[i] = f32_from_f64(y);
    a.fz[i] = f32_from_f64(z);
    a.ja[i] = sqrt_obs(dot3(x, y, z, x, y, z));
  }
  __syncwarp(gm);
  double sum_abs = 0.0;
  for (int i = 0; i < n; ++i) sum_abs += a.ja[i];
  const float sum_absf = f32_from_f64(sum_abs);

  // ---- thrust
  double thrust = 1.0, ax = 0.0, ay = 0.0, az = 0.0;
  bool decided = false;
  if (n == 2) {
    const double inv_l = 1.0 / a.ja[0];
    ax = a.j[1][0] * inv_l;
    ay = a.j[2][0] * inv_l;
    az = a.j[3][0] * inv_l;
    decided = true;
  } else {
    static_assert(MAXJ < 64, "a partition is a word");
    Top2 top;
    const unsigned long long full = (1ull << n) - 1ull;
    PairWalk w;
    for (w.start(n, sub); w.valid(n); w.next<L>(n)) {
      const int j = w.j, k = w.k();
      const float nx = crossf(a.fy[j], a.fz[k], a.fz[j], a.fy[k]);
      const float ny = crossf(a.fz[j], a.fx[k], a.fx[j], a.fz[k]);
      const float nz = crossf(a.fx[j], a.fy[k], a.fy[j], a.fx[k]);
      if (nx == 0.0f && ny == 0.0f && nz == 0.0f) continue;
      float px = 0.0f, py = 0.0f, pz = 0.0f;
      unsigned long long mask = 0ull;
      for (int i = 0; i < n; ++i) {
        if (i == j || i == k) continue;
        if (dot3f(a.fx[i], a.fy[i], a.fz[i], nx, ny, nz) >= 0.0f) {
          px += a.fx[i];
          py += a.fy[i];
          pz += a.fz[i];
          mask |= 1ull << i;
        } else {
          px -= a.fx[i];
          py -= a.fy[i];
          pz -= a.fz[i];
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const bool pj = !(c & 2), pk = !(c & 1);
        const float cx = px + (pj ? a.fx[j] : -a.fx[j]) + (pk ? a.fx[k] : -a.fx[k]);
        const float cy = py + (pj ? a.fy[j] : -a.fy[j]) + (pk ? a.fy[k] : -a.fy[k]);
        const float cz = pz + (pj ? a.fz[j] : -a.fz[j]) + (pk ? a.fz[k] : -a.fz[k]);
        unsigned long long m = mask | (pj ? 1ull << j : 0ull) | (pk ? 1ull << k : 0ull);
        if (m & 1ull) m = ~m & full;
        top.add(dot3f(cx, cy, cz, cx, cy, cz), m);
      }
    }
    // The top two distinct partitions of the union: each lane's two entries
    // added to the other's (the best score of every partition reaches the
    // merged pair; only which of two equal scores is first can depend on
    // the order, and equal scores leave the search to the exact FP64 pass).
#pragma unroll
    for (int off = 1; off < L; off <<= 1) {
      const float s1 = __shfl_xor_sync(gm, top.s1, off), s2 = __shfl_xor_sync(gm, top.s2, off);
      const unsigned long long m1 = __shfl_xor_sync(gm, top.m1, off), m2 = __shfl_xor_sync(gm, top.m2, off);
      top.add(s1, m1);
      top.add(s2, m2);
    }
    const float margin = 8.0f * static_cast<float>(n + 2) * 6.0e-8f * sum_absf * sum_absf;
    if (top.s1 >= 0.0f && top.s2 < top.s1 - margin) {
      // a component per lane, each summed in the serial order
      double sum = 0.0;
      const int c = 1 + min(sub, 2);
      for (int i = 0; i < n; ++i) sum = fma(((top.m1 >> i) & 1ull) ? 1.0 : -1.0, a.j[c][i], sum);
      const int g0 = static_cast<int>(threadIdx.x & 31u) - sub;
      const double px = __shfl_sync(gm, sum, g0), py = __shfl_sync(gm, sum, g0 + 1);
      const double pz = __shfl_sync(gm, sum, g0 + 2);
      const double l = sqrt_obs(dot3(px, py, pz, px, py, pz)), inv_l = 1.0 / l;
      thrust = l / sum_abs;
      ax = px * inv_l;
      ay = py * inv_l;
      az = pz * inv_l;
      decided = true;
    }
  }
  if (!decided) {
    if (sub == 0) atomicAdd(&E.counters[4], 1ull);  // thrust decided by the exact FP64 search
    thrust = thrust_fp64_group<MAXJ, L>(n, a, sum_abs, sub, gm, ax, ay, az);
  }
  // Hemispheres: every parton's side and |p x n_T| on a lane of its own, the
  // sums one per lane in the serial order.
  for (int i = sub; i < n; i += L) {
    const double x = a.j[1][i], y = a.j[2][i], z = a.j[3][i];
    const long long pn = __double_as_longlong(dot3(x, y, z, ax, ay, az));
    a.plus[i] = pn >= 0 || pn == static_cast<long long>(0x8000000000000000ull);
    const double cx = cross(y, az, z, ay), cy = cross(z, ax, x, az), cz = cross(x, ay, y, ax);
    a.pt[i] = sqrt_obs(dot3(cx, cy, cz, cx, cy, cz));
  }
  __syncwarp(gm);
  for (int c = sub; c < 5; c += L) {
    const double* v = c < 4 ? a.j[c] : a.pt;
    double plus = 0.0, minus = 0.0;
    for (int i = 0; i < n; ++i) {
      const bool p = a.plus[i] != 0;
      const double sum = (p ? plus : minus) + v[i];
      plus = p ? sum : plus;
      minus = p ? minus : sum;
    }
    a.sums[0][c] = plus;
    a.sums[1][c] = minus;
  }
  __syncwarp(gm);
  if (sub == 0) {
    const double mp = mass2(a.sums[0]);
    const double mm = mass2(a.sums[1]);
    E.obs[4 * E.stride + ev] = 1.0 - thrust;
    E.obs[5 * E.stride + ev] = fmax(mp, mm) * P.inv_s;
    const double inv_2sum = 0.5 / sum_abs;
    const double bp = a.sums[0][4] * inv_2sum, bm = a.sums[1][4] * inv_2sum;
    E.obs[6 * E.stride + ev] = bp + bm;
    E.obs[7 * E.stride + ev] = fmax(bp, bm);
  }

  // ---- Durham (E-scheme)
  __syncwarp(gm);  // every lane has read the FP32 momenta
  for (int i = sub; i < n; i += L) {
    const float e = f32_from_f64(a.j[0][i]);
    a.fe2[i] = e * e;
    const float r = rsqrtf(dot3f(a.fx[i], a.fy[i], a.fz[i], a.fx[i], a.fy[i], a.fz[i]));
    a.fx[i] *= r;
    a.fy[i] *= r;
    a.fz[i] *= r;
  }
  __syncwarp(gm);
  double yres[4] = {-1.0, -1.0, -1.0, -1.0};
  auto y_exact = [&](int i, int j) {
    const double cosij = dot3(a.j[1][i], a.j[2][i], a.j[3][i], a.j[1][j], a.j[2][j], a.j[3][j]) / (a.ja[i] * a.ja[j]);
    return 2.0 * fmin(a.j[0][i] * a.j[0][i], a.j[0][j] * a.j[0][j]) * (1.0 - cosij) * P.inv_s;
  };
  auto bounds = [&](int i, int j, float& y, float& rel) {
    const float dx = a.fx[i] - a.fx[j], dy = a.fy[i] - a.fy[j], dz = a.fz[i] - a.fz[j];
    const float d = dot3f(dx, dy, dz, dx, dy, dz);
    y = fminf(a.fe2[i], a.fe2[j]) * d;
    rel = 4.0e-6f + 1.0e-6f * rsqrtf(fmaxf(d, 1e-30f));
  };
  for (int m = n; m > 2; --m) {  // y of the last two jets is not recorded
    // pass 1: the smallest FP32 upper bound, the first pair on ties
    float ubest = INFINITY;
    int up = 0x7fffffff, ui = 0, uj = 1;
    PairWalk w;
    for (w.start(m, sub); w.valid(m); w.next<L>(m)) {
      float y, rel;
      bounds(w.j, w.k(), y, rel);
      const float ub = fmaf(y, 1.0f + rel, 1e-30f);
      if (ub < ubest) {
        ubest = ub;
        up = w.p;
        ui = w.j;
        uj = w.k();
      }
    }
#pragma unroll
    for (int off = 1; off < L; off <<= 1) {
      const float ou = __shfl_xor_sync(gm, ubest, off);
      const int op = __shfl_xor_sync(gm, up, off), oi = __shfl_xor_sync(gm, ui, off);
      const int oj = __shfl_xor_sync(gm, uj, off);
      if (ou < ubest || (ou == ubest && op < up)) {
        ubest = ou;
        up = op;
        ui = oi;
        uj = oj;
      }
    }
    // pass 2: the pairs whose lower bound reaches it
    int n_cand = 0;
    for (w.start(m, sub); w.valid(m); w.next<L>(m)) {
      float y, rel;
      bounds(w.j, w.k(), y, rel);
      n_cand += y * (1.0f - rel) <= ubest ? 1 : 0;
    }
#pragma unroll
    for (int off = 1; off < L; off <<= 1) n_cand += __shfl_xor_sync(gm, n_cand, off);
    double ymin = 0.0;
    int bi = ui, bj = uj;
    if (n_cand == 1) {
      if (m <= 6) ymin = y_exact(ui, uj);  // the merges that are recorded
    } else {
      if (sub == 0) atomicAdd(&E.counters[5], 1ull);  // merges with several FP64 candidates
      int bp_ = 0x7fffffff;
      ymin = INFINITY;
      for (w.start(m, sub); w.valid(m); w.next<L>(m)) {
        float y, rel;
        bounds(w.j, w.k(), y, rel);
        if (y * (1.0f - rel) > ubest) continue;
        const double yy = y_exact(w.j, w.k());
        if (bp_ == 0x7fffffff || yy < ymin) {
          ymin = yy;
          bp_ = w.p;
          bi = w.j;
          bj = w.k();
        }
      }
#pragma unroll
      for (int off = 1; off < L; off <<= 1) {
        const double oy = __shfl_xor_sync(gm, ymin, off);
        const int op = __shfl_xor_sync(gm, bp_, off), oi = __shfl_xor_sync(gm, bi, off);
        const int oj = __shfl_xor_sync(gm, bj, off);
        // lanes without a candidate hold position 0x7fffffff
        if (op != 0x7fffffff && (bp_ == 0x7fffffff || oy < ymin || (oy == ymin && op < bp_))) {
          ymin = oy;
          bp_ = op;
          bi = oi;
          bj = oj;
        }
      }
    }
    if (m <= 6) yres[m - 3] = ymin;
    if (m == 3) break;
    __syncwarp(gm);  // every lane is done reading the jets of this merge
    if (sub < 4) {  // a component per lane (L >= 4)
      a.j[sub][bi] += a.j[sub][bj];
      a.j[sub][bj] = a.j[sub][m - 1];
    }
    __syncwarp(gm);
    if (sub == 0) {
      const double jx = a.j[1][bi], jy = a.j[2][bi], jz = a.j[3][bi];
      a.ja[bj] = a.ja[m - 1];
      a.ja[bi] = sqrt_obs(dot3(jx, jy, jz, jx, jy, jz));
      a.fe2[bj] = a.fe2[m - 1];
      a.fx[bj] = a.fx[m - 1];
      a.fy[bj] = a.fy[m - 1];
      a.fz[bj] = a.fz[m - 1];
      const float e = f32_from_f64(a.j[0][bi]);
      a.fe2[bi] = e * e;
      const float x = f32_from_f64(jx), y = f32_from_f64(jy), z = f32_from_f64(jz);
      const float r = rsqrtf(dot3f(x, y, z, x, y, z));
      a.fx[bi] = x * r;
      a.fy[bi] = y * r;
      a.fz[bi] = z * r;
    }
    __syncwarp(gm);
  }
  if (sub == 0)
    for (int h = 0; h < 4; ++h) E.obs[h * E.stride + ev] = yres[h];
}

// ------------------------------------------------- a warp per large event
// The event of a warp in shared memory.  f: FP32 unit directions, with |p| in
// the thrust search and E^2 in the clustering.  Durham's nearest neighbours: jet
// r's smallest upper bound ub of the distance to another jet (near, with
// lower bound lb) and a lower bound lb2 of all others: the smallest of theirs
// (near2's), or no more than that once near2 is gone (near2 = kGone).
template <int MAXJ>
struct WarpEvent {
  double j[4][MAXJ];  // E, px, py, pz
  float4 f[MAXJ];
  float ub[MAXJ], lb[MAXJ], lb2[MAXJ];
  uint8_t near[MAXJ], near2[MAXJ];
  uint32_t full[MAXJ / 32], lengthy[MAXJ / 32];  // partitions' bits in use, and those of partons of some length
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// A partition of up to 32 W partons as sign bits (set: the minus side), 32 a
// word (side_bit).
template <int W>
struct Partition {
  uint32_t w[W];
  __device__ __forceinline__ bool operator==(const Partition& o) const {
    uint32_t d = 0u;
#pragma unroll
    for (int c = 0; c < W; ++c) d |= w[c] ^ o.w[c];
    return d == 0u;
  }
};
// The kTop best distinct partitions by score, in no order; `least` is the
// smallest of their scores.
constexpr int kTop = 4;
template <int W>
struct TopPartitions {
  float s[kTop];
  Partition<W> m[kTop];
  float least = -1.0f;
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int t = 0; t < kTop; ++t) {
      s[t] = -1.0f;
#pragma unroll
      for (int c = 0; c < W; ++c) m[t].w[c] = 0u;
    }
  }
  // (a score at or below the least changes nothing)
  __device__ __forceinline__ void add(float v, const Partition<W>& p) {
    int at = -1, low = 0;
#pragma unroll
    for (int t = 0; t < kTop; ++t) {
      if (s[t] >= 0.0f && m[t] == p) at = t;
      if (s[t] == least) low = t;
    }
    const int to = at >= 0 ? at : low;
    least = INFINITY;
#pragma unroll
    for (int t = 0; t < kTop; ++t) {
      if (t == to) {
        s[t] = at >= 0 ? fmaxf(s[t], v) : v;
        m[t] = p;
      }
      least = fminf(least, s[t]);
    }
  }
};

// Bit of parton i in word c of a partition of n partons.  The pairs' loop
// collects two bits a parton, the last one's lowest, the first 16 of a word
// apart from its second 16: the first have the odd bits, the second the even.
__device__ __forceinline__ uint32_t side_bit(int n, int i, int c) {
  const int first = i & ~15, last = min(n, first + 16) - 1;
  return i >> 5 == c ? 1u << (2 * (last - i) + ((i & 16) == 0 ? 1 : 0)) : 0u;
}

// The sides of a pair's plane: the other partons' partition and their signed
// sum (the pair's own two in neither).
template <int W>
struct Sides {
  Partition<W> m;
  float x, y, z;
};

// FP32 sides.  A product of the unit direction u_i with the normal u_j x u_k
// is off by up to 6.6e-7: the directions' components by 2^-23 each (three
// vectors, 3.6e-7), the normal's by 2^-23 (1.2e-7), the product's rounding by
// 3 x 2^-24 (1.8e-7).  Normals are scaled by 2^21, so that a product within
// 2^-20 of zero, whose sign is in doubt, is one below 2: the top bit of its
// exponent is clear.  The two top bits of every product are collected, the
// sign and whether it is certain, by one shift as the sign alone would be.
// Returns whether every parton's of some length is certain, the pair's own two
// excepted.
constexpr float kNormalScale = 2097152.0f;  // 2^21
template <int MAXJ>
__device__ __forceinline__ bool sides_fp32(const WarpEvent<MAXJ>& a, int n, int j, int k, Sides<MAXJ / 32>& o) {
  const float4 uj = a.f[j], uk = a.f[k];
  const float nx = kNormalScale * crossf(uj.y, uk.z, uj.z, uk.y);
  const float ny = kNormalScale * crossf(uj.z, uk.x, uj.x, uk.z);
  const float nz = kNormalScale * crossf(uj.x, uk.y, uj.y, uk.x);
  const uint32_t jbit = side_bit(n, j, j >> 5), kbit = side_bit(n, k, k >> 5);
  o.x = o.y = o.z = 0.0f;
  uint32_t own_j = 0u, own_k = 0u, doubt = 0u;
#pragma unroll
  for (int c = 0; c < MAXJ / 32; ++c) {
    o.m.w[c] = 0u;
    if (32 * c >= n) continue;
    uint32_t odd = 0u, even = 0u;
    const auto take = [&](int i, uint32_t& bits) {
      const float4 u = a.f[i];
      const uint32_t s = __float_as_uint(dot3f(u.x, u.y, u.z, nx, ny, nz));
      const float w = __uint_as_float((s & 0x80000000u) | __float_as_uint(u.w));
      o.x = fmaf(w, u.x, o.x);
      o.y = fmaf(w, u.y, o.y);
      o.z = fmaf(w, u.z, o.z);
      bits = __funnelshift_l(s, bits, 2);
    };
    const int n_odd = min(n - 32 * c, 16), n_even = min(max(n - 32 * c - 16, 0), 16);
    int t = 0;
#pragma unroll 1
    for (; t < n_even; ++t) {
      take(32 * c + t, odd);
      take(32 * c + 16 + t, even);
    }
#pragma unroll 1
    for (; t < n_odd; ++t) take(32 * c + t, odd);
    const uint32_t sign = (odd & 0xaaaaaaaau) | ((even & 0xaaaaaaaau) >> 1);
    const uint32_t known = ((odd & 0x55555555u) << 1) | (even & 0x55555555u);
    const uint32_t jb = j >> 5 == c ? jbit : 0u, kb = k >> 5 == c ? kbit : 0u;
    doubt |= a.lengthy[c] & ~(known | jb | kb);
    own_j |= sign & jb;
    own_k |= sign & kb;
    o.m.w[c] = sign & ~(jb | kb);
  }
  // without the pair itself
  const float wj = own_j ? uj.w : -uj.w, wk = own_k ? uk.w : -uk.w;
  o.x = fmaf(wk, uk.x, fmaf(wj, uj.x, o.x));
  o.y = fmaf(wk, uk.y, fmaf(wj, uj.y, o.y));
  o.z = fmaf(wk, uk.z, fmaf(wj, uj.z, o.z));
  return doubt == 0u;
}

// FP64 sides, with the exact search's formulas, by the whole warp; false where
// the pair spans no plane.  About one pair in 10^4 of an isotropic event comes
// here, every pair of a planar one.
template <int MAXJ>
__device__ __noinline__ bool sides_fp64(const WarpEvent<MAXJ>& a, int n, int j, int k, int lane, Sides<MAXJ / 32>& o) {
  const double nx = cross(a.j[2][j], a.j[3][k], a.j[3][j], a.j[2][k]);
  const double ny = cross(a.j[3][j], a.j[1][k], a.j[1][j], a.j[3][k]);
  const double nz = cross(a.j[1][j], a.j[2][k], a.j[2][j], a.j[1][k]);
  if (nx == 0.0 && ny == 0.0 && nz == 0.0) return false;
  float x = 0.0f, y = 0.0f, z = 0.0f;
#pragma unroll
  for (int c = 0; c < MAXJ / 32; ++c) {
    const int i = 32 * c + lane;
    uint32_t bit = 0u;
    if (i < n && i != j && i != k) {
      const bool plus = dot3(a.j[1][i], a.j[2][i], a.j[3][i], nx, ny, nz) >= 0.0;
      const float4 u = a.f[i];
      const float w = plus ? u.w : -u.w;
      x = fmaf(w, u.x, x);
      y = fmaf(w, u.y, y);
      z = fmaf(w, u.z, z);
      bit = plus ? 0u : side_bit(n, i, c);
    }
    o.m.w[c] = __reduce_or_sync(0xffffffffu, bit);
  }
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    x += __shfl_xor_sync(0xffffffffu, x, off);
    y += __shfl_xor_sync(0xffffffffu, y, off);
    z += __shfl_xor_sync(0xffffffffu, z, off);
  }
  o.x = x;
  o.y = y;
  o.z = z;
  return true;
}

// FP32 bounds of the distance of jets a and b (unit directions, E^2 in w):
// per-pair relative error 4e-6 + 1e-6 / |u_a - u_b|.
__device__ __forceinline__ void pair_bounds(const float4& a, const float4& b, float& ub, float& lb) {
  const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
  const float d = dot3f(dx, dy, dz, dx, dy, dz);
  const float y = fminf(a.w, b.w) * d;
  const float rel = 4.0e-6f + 1.0e-6f * rsqrtf(fmaxf(d, 1e-30f));
  ub = fmaf(y, 1.0f + rel, 1e-30f);
  lb = y * (1.0f - rel);
}

// A row of the nearest-neighbour table.
constexpr int kGone = 255;
struct Row {
  float ub, lb, lb2;
  int near, near2;
  __device__ __forceinline__ void clear() {
    ub = lb = lb2 = INFINITY;
    near = near2 = kGone;
  }
  __device__ __forceinline__ void add(float u, float l, int k) {
    if (u < ub) {
      if (lb < lb2) {
        lb2 = lb;
        near2 = near;
      }
      ub = u;
      lb = l;
      near = k;
    } else if (l < lb2) {
      lb2 = l;
      near2 = k;
    }
  }
};
template <int MAXJ>
__device__ __forceinline__ Row load_row(const WarpEvent<MAXJ>& a, int r) {
  return Row{a.ub[r], a.lb[r], a.lb2[r], a.near[r], a.near2[r]};
}
template <int MAXJ>
__device__ __forceinline__ void store_row(WarpEvent<MAXJ>& a, int r, const Row& row) {
  a.ub[r] = row.ub;
  a.lb[r] = row.lb;
  a.lb2[r] = row.lb2;
  a.near[r] = static_cast<uint8_t>(row.near);
  a.near2[r] = static_cast<uint8_t>(row.near2);
}

// |p| of jet i.
template <int MAXJ>
__device__ __forceinline__ double jet_length(const WarpEvent<MAXJ>& a, int i) {
  return sqrt_obs(dot3(a.j[1][i], a.j[2][i], a.j[3][i], a.j[1][i], a.j[2][i], a.j[3][i]));
}
// y of jets i and k with the oracle's FP64 formula.
template <int MAXJ>
__device__ __forceinline__ double jet_distance(const WarpEvent<MAXJ>& a, int i, int k, double inv_s) {
  const double cosik = dot3(a.j[1][i], a.j[2][i], a.j[3][i], a.j[1][k], a.j[2][k], a.j[3][k]) /
                       (jet_length(a, i) * jet_length(a, k));
  return 2.0 * fmin(a.j[0][i] * a.j[0][i], a.j[0][k] * a.j[0][k]) * (1.0 - cosik) * inv_s;
}

// thrust_fp64 over the warp (see thrust_fp64_group).
template <int MAXJ>
__device__ __noinline__ double thrust_fp64_warp(int n, const WarpEvent<MAXJ>& a, double sum_abs, int lane, double& ax,
                                                double& ay, double& az) {
  double best2 = -1.0, bx = 0.0, by = 0.0, bz = 0.0;
  int bidx = 0x7fffffff;
  PairWalk w;
  for (w.start(n, lane); w.valid(n); w.next<32>(n)) {
    const int j = w.j, k = w.k();
    const double nx = cross(a.j[2][j], a.j[3][k], a.j[3][j], a.j[2][k]);
    const double ny = cross(a.j[3][j], a.j[1][k], a.j[1][j], a.j[3][k]);
    const double nz = cross(a.j[1][j], a.j[2][k], a.j[2][j], a.j[1][k]);
    if (nx == 0.0 && ny == 0.0 && nz == 0.0) continue;
    double px = 0.0, py = 0.0, pz = 0.0;
    for (int i = 0; i < n; ++i) {
      if (i == j || i == k) continue;
      const double sg = dot3(a.j[1][i], a.j[2][i], a.j[3][i], nx, ny, nz) >= 0.0 ? 1.0 : -1.0;
      px = fma(sg, a.j[1][i], px);
      py = fma(sg, a.j[2][i], py);
      pz = fma(sg, a.j[3][i], pz);
    }
    for (int c = 0; c < 4; ++c) {
      const double fj = (c & 2) ? -1.0 : 1.0, fk = (c & 1) ? -1.0 : 1.0;
      const double cx = fma(fk, a.j[1][k], fma(fj, a.j[1][j], px));
      const double cy = fma(fk, a.j[2][k], fma(fj, a.j[2][j], py));
      const double cz = fma(fk, a.j[3][k], fma(fj, a.j[3][j], pz));
      const double c2 = dot3(cx, cy, cz, cx, cy, cz);
      if (c2 > best2) {  // within a lane the positions rise: the first wins ties
        best2 = c2;
        bidx = 4 * w.p + c;
        bx = cx;
        by = cy;
        bz = cz;
      }
    }
  }
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const double o2 = __shfl_xor_sync(0xffffffffu, best2, off);
    const int oi = __shfl_xor_sync(0xffffffffu, bidx, off);
    const double ox = __shfl_xor_sync(0xffffffffu, bx, off), oy = __shfl_xor_sync(0xffffffffu, by, off);
    const double oz = __shfl_xor_sync(0xffffffffu, bz, off);
    if (o2 > best2 || (o2 == best2 && oi < bidx)) {
      best2 = o2;
      bidx = oi;
      bx = ox;
      by = oy;
      bz = oz;
    }
  }
  if (best2 < 0.0) {  // collinear: T = 1 along the first momentum
    const double l = jet_length(a, 0);
    ax = a.j[1][0] / l;
    ay = a.j[2][0] / l;
    az = a.j[3][0] / l;
    return 1.0;
  }
  const double l = sqrt_obs(best2), inv_l = 1.0 / l;
  ax = bx * inv_l;
  ay = by * inv_l;
  az = bz * inv_l;
  return l / sum_abs;
}

// The observables of one event of more than 16 partons, by a warp.
//
// Thrust: the lanes take the pairs; a pair's partition is built from the
// signs of the other momenta's products with its normal without a branch (the
// pair's own two, whose products are rounding, are taken out of the sum
// afterwards), and again by the warp in FP64 where a sign is in doubt: of 65
// momenta that lie 10^-8 out of a plane or of three directions, FP32 signs
// alone gave another axis than the exact search.  With the four best distinct
// partitions known, those within the FP32 error of the best are compared in
// FP64, unless the fourth is one of them (with many partons the best two often
// are: one event in fifty of 17 .. 80 partons was left to the exact search,
// which takes half a millisecond); the winner must also be the one its own
// axis defines, which the longest one is.
//
// Durham: a merge changes the distances to one jet only, so every jet keeps
// its nearest neighbour and a lower bound of the others' (Row); a merge renews
// the rows that pointed at the two merged jets, by the whole warp, and offers
// the new jet to the others.  A row whose second neighbour is gone keeps the
// old bound, and is renewed only where that bound is too low to decide.  One jet pair decides a merge from its
// FP32 bounds as before; y in FP64 is only formed for the four merges that
// are recorded.
//
// Bound by FP32 issue in the thrust pairs (n^3 / 2 products, eight
// instructions each).  20 000 RAMBO events of 17 .. 80 partons: 25.3 -> 3.1 ms
// against every merge searching all its pairs twice, events beyond 64 partons
// searched in FP64, and two blocks per SM with a fixed share of the events
// each (with these in place: 7.3 ms with two partitions kept and every row that
// pointed at a merged jet renewed, 4.8 ms with fixed shares); 3.2 ms with the
// signs made certain (3.4 with the two halves of a word in loops of their own).
template <int MAXJ>
__device__ void event_shapes_warp(const DevParams& P0, const Events& E, int64_t ev, int n, WarpEvent<MAXJ>& a, int lane) {
  constexpr int W = MAXJ / 32;
  const DevParams& P = params_of_event(P0, E, ev);
  double sum_abs = 0.0;
  for (int i = lane; i < n; i += 32) {
    const size_t at = E.at(i, ev);
    const double x = E.px[at], y = E.py[at], z = E.pz[at];
    a.j[0][i] = E.e[at];
    a.j[1][i] = x;
    a.j[2][i] = y;
    a.j[3][i] = z;
    const double length = sqrt_obs(dot3(x, y, z, x, y, z));
    sum_abs += length;
    const float fx = f32_from_f64(x), fy = f32_from_f64(y), fz = f32_from_f64(z);
    const float l2 = dot3f(fx, fy, fz, fx, fy, fz), r = rsqrtf(l2);
    // (of no length in single precision: on either side, and no part of a sum)
    a.f[i] = l2 == 0.0f ? make_float4(0.0f, 0.0f, 0.0f, 0.0f) : make_float4(fx * r, fy * r, fz * r, f32_from_f64(length));
  }
  sum_abs = warp_sum(sum_abs);
  const float sum_absf = f32_from_f64(sum_abs);
  __syncwarp();

  // ---- thrust
  TopPartitions<W> top;
  top.clear();
#pragma unroll
  for (int c = 0; c < W; ++c) {
    const int i = 32 * c + lane;
    const uint32_t bit = i < n ? side_bit(n, i, c) : 0u;
    const uint32_t all = __reduce_or_sync(0xffffffffu, bit);
    const uint32_t some = __reduce_or_sync(0xffffffffu, i < n && a.f[i].w != 0.0f ? bit : 0u);
    if (lane == 0) {
      a.full[c] = all;
      a.lengthy[c] = some;
    }
  }
  __syncwarp();
  PairWalk pw;
  pw.start(n, lane);
#pragma unroll 1
  for (;;) {
    bool has = pw.valid(n);
    if (!__any_sync(0xffffffffu, has)) break;
    const int j = has ? pw.j : 0, k = has ? pw.k() : 1;
    Sides<W> sides;
    const bool certain = sides_fp32<MAXJ>(a, n, j, k, sides);
    unsigned doubt = __ballot_sync(0xffffffffu, has && !certain);
#pragma unroll 1
    while (doubt != 0u) {
      const int src = __ffs(doubt) - 1;
      doubt &= doubt - 1u;
      Sides<W> exact;
      const bool plane = sides_fp64<MAXJ>(a, n, __shfl_sync(0xffffffffu, j, src), __shfl_sync(0xffffffffu, k, src), lane, exact);
      if (lane == src) {
        has = plane;
        sides.x = exact.x;
        sides.y = exact.y;
        sides.z = exact.z;
        sides.m = exact.m;
      }
    }
    if (has) {
      const float4 uj = a.f[j], uk = a.f[k];
      const uint32_t jbit = side_bit(n, j, j >> 5), kbit = side_bit(n, k, k >> 5), bit0 = side_bit(n, 0, 0);
#pragma unroll 1
      for (int c4 = 0; c4 < 4; ++c4) {
        const float wj = (c4 & 2) ? -uj.w : uj.w, wk = (c4 & 1) ? -uk.w : uk.w;
        const float cx = fmaf(wk, uk.x, fmaf(wj, uj.x, sides.x));
        const float cy = fmaf(wk, uk.y, fmaf(wj, uj.y, sides.y));
        const float cz = fmaf(wk, uk.z, fmaf(wj, uj.z, sides.z));
        const float score = dot3f(cx, cy, cz, cx, cy, cz);
        if (score <= top.least) continue;
        Partition<W> t;
#pragma unroll
        for (int c = 0; c < W; ++c)
          t.w[c] = sides.m.w[c] | ((c4 & 2) && j >> 5 == c ? jbit : 0u) | ((c4 & 1) && k >> 5 == c ? kbit : 0u);
        if (t.w[0] & bit0) {  // a partition and its complement are one candidate
#pragma unroll
          for (int c = 0; c < W; ++c) t.w[c] = ~t.w[c] & a.full[c];
        }
        top.add(score, t);
      }
    }
    pw.next<32>(n);
  }
#pragma unroll 1
  for (int off = 1; off < 32; off <<= 1) {
    float os[kTop];
    Partition<W> om[kTop];
#pragma unroll
    for (int t = 0; t < kTop; ++t) {  // all before the first addition
      os[t] = __shfl_xor_sync(0xffffffffu, top.s[t], off);
#pragma unroll
      for (int c = 0; c < W; ++c) om[t].w[c] = __shfl_xor_sync(0xffffffffu, top.m[t].w[c], off);
    }
#pragma unroll
    for (int t = 0; t < kTop; ++t)
      if (os[t] > top.least) top.add(os[t], om[t]);
  }
  float best = top.s[0];
#pragma unroll
  for (int t = 1; t < kTop; ++t) best = fmaxf(best, top.s[t]);
  const float margin = 8.0f * static_cast<float>(n + 2) * 6.0e-8f * sum_absf * sum_absf;
  double thrust = 1.0, ax = 0.0, ay = 0.0, az = 0.0;
  bool decided = best >= 0.0f && top.least < best - margin;
  if (decided) {
    // the partitions within the error of the best, in FP64: the longest, if
    // it is longer than the others by more than their rounding
    double l2 = -1.0, next2 = -1.0;
    Partition<W> won{};
#pragma unroll 1
    for (int t = 0; t < kTop; ++t) {
      Partition<W> m = top.m[0];
      float v = top.s[0];
#pragma unroll
      for (int u = 1; u < kTop; ++u)
        if (t == u) {
          m = top.m[u];
          v = top.s[u];
        }
      // every lane holds the same partitions, but not in the same places:
      // lane 0's
      v = __shfl_sync(0xffffffffu, v, 0);
#pragma unroll
      for (int c = 0; c < W; ++c) m.w[c] = __shfl_sync(0xffffffffu, m.w[c], 0);
      if (v < best - margin) continue;
      double px = 0.0, py = 0.0, pz = 0.0;
      for (int i = lane; i < n; i += 32) {
        uint32_t minus = 0u;
#pragma unroll
        for (int c = 0; c < W; ++c) minus |= m.w[c] & side_bit(n, i, c);
        const double sg = minus ? -1.0 : 1.0;
        px = fma(sg, a.j[1][i], px);
        py = fma(sg, a.j[2][i], py);
        pz = fma(sg, a.j[3][i], pz);
      }
      px = warp_sum(px);
      py = warp_sum(py);
      pz = warp_sum(pz);
      const double c2 = dot3(px, py, pz, px, py, pz);
      if (c2 > l2) {
        next2 = l2;
        l2 = c2;
        won = m;
        ax = px;
        ay = py;
        az = pz;
      } else {
        next2 = fmax(next2, c2);
      }
    }
    decided = next2 < l2 * (1.0 - 1e-12);
    const double l = sqrt_obs(l2), inv_l = 1.0 / l;
    thrust = l / sum_abs;
    ax *= inv_l;
    ay *= inv_l;
    az *= inv_l;
    // every parton on the side of the axis its sign says
    for (int i = lane; i < n; i += 32) {
      uint32_t minus = 0u;
#pragma unroll
      for (int c = 0; c < W; ++c) minus |= won.w[c] & side_bit(n, i, c);
      const double d = dot3(a.j[1][i], a.j[2][i], a.j[3][i], ax, ay, az);
      decided = decided && (minus ? d <= 0.0 : d >= 0.0);
    }
    decided = __all_sync(0xffffffffu, decided);
  }
  if (!decided) {
    if (lane == 0) atomicAdd(&E.counters[4], 1ull);  // thrust decided by the exact FP64 search
    thrust = thrust_fp64_warp<MAXJ>(n, a, sum_abs, lane, ax, ay, az);
  }
  // Hemispheres: heavy-jet mass and jet broadenings.
  double hp[4] = {0, 0, 0, 0}, hm[4] = {0, 0, 0, 0};
  double bp = 0.0, bm = 0.0;
  for (int i = lane; i < n; i += 32) {
    const double x = a.j[1][i], y = a.j[2][i], z = a.j[3][i];
    const long long pn = __double_as_longlong(dot3(x, y, z, ax, ay, az));
    const bool plus = pn >= 0 || pn == static_cast<long long>(0x8000000000000000ull);
    const double cx = cross(y, az, z, ay), cy = cross(z, ax, x, az), cz = cross(x, ay, y, ax);
    const double pt = sqrt_obs(dot3(cx, cy, cz, cx, cy, cz));
    double* h = plus ? hp : hm;
    h[0] += a.j[0][i];
    h[1] += x;
    h[2] += y;
    h[3] += z;
    if (plus) {
      bp += pt;
    } else {
      bm += pt;
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    hp[c] = warp_sum(hp[c]);
    hm[c] = warp_sum(hm[c]);
  }
  bp = warp_sum(bp);
  bm = warp_sum(bm);
  if (lane == 0) {
    const double mp = mass2(hp), mm = mass2(hm);
    E.obs[4 * E.stride + ev] = 1.0 - thrust;
    E.obs[5 * E.stride + ev] = fmax(mp, mm) * P.inv_s;
    const double inv_2sum = 0.5 / sum_abs;
    bp *= inv_2sum;
    bm *= inv_2sum;
    E.obs[6 * E.stride + ev] = bp + bm;
    E.obs[7 * E.stride + ev] = fmax(bp, bm);
  }

  // ---- Durham (E-scheme)
  const auto direction = [&](int i) {
    const float e = f32_from_f64(a.j[0][i]);
    const float x = f32_from_f64(a.j[1][i]), y = f32_from_f64(a.j[2][i]), z = f32_from_f64(a.j[3][i]);
    const float r = rsqrtf(dot3f(x, y, z, x, y, z));
    return make_float4(x * r, y * r, z * r, e * e);
  };
  __syncwarp();  // every lane is done with the FP32 momenta
  for (int i = lane; i < n; i += 32) a.f[i] = direction(i);
  __syncwarp();
  for (int r = lane; r < n; r += 32) {
    Row row;
    row.clear();
    const float4 fr = a.f[r];
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
      if (k == r) continue;
      float u, l;
      pair_bounds(fr, a.f[k], u, l);
      row.add(u, l, k);
    }
    store_row(a, r, row);
  }
  // Row t anew from the jets 0 .. m - 1, by the whole warp.
  const auto renew_row = [&](int t, int m) {
    const float4 ft = a.f[t];
    Row row;
    row.clear();
    for (int k = lane; k < m; k += 32) {
      if (k == t) continue;
      float u, l;
      pair_bounds(ft, a.f[k], u, l);
      row.add(u, l, k);
    }
#pragma unroll 1
    for (int off = 1; off < 32; off <<= 1) {
      const float ou = __shfl_xor_sync(0xffffffffu, row.ub, off), ol = __shfl_xor_sync(0xffffffffu, row.lb, off);
      const float o2 = __shfl_xor_sync(0xffffffffu, row.lb2, off);
      const int both = __shfl_xor_sync(0xffffffffu, row.near | (row.near2 << 8), off);
      const int on = both & 255, on2 = both >> 8;
      // the better nearest stays; the other's and both seconds compete
      const bool theirs = ou < row.ub || (ou == row.ub && on < row.near);
      float c1 = theirs ? row.lb : ol;
      int k1 = theirs ? row.near : on;
      if (theirs) {
        row.ub = ou;
        row.lb = ol;
        row.near = on;
      }
      if (o2 < c1) {
        c1 = o2;
        k1 = on2;
      }
      if (c1 < row.lb2) {
        row.lb2 = c1;
        row.near2 = k1;
      }
    }
    if (lane == 0) store_row(a, t, row);
  };
  double yres[4] = {-1.0, -1.0, -1.0, -1.0};
#pragma unroll 1
  for (int m = n; m > 2; --m) {  // y of the last two jets is not recorded
    __syncwarp();
    // the smallest upper bound and its pair
    float ubest = INFINITY;
    int br = 0;
    for (int r = lane; r < m; r += 32)
      if (a.ub[r] < ubest) {
        ubest = a.ub[r];
        br = r;
      }
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float ou = __shfl_xor_sync(0xffffffffu, ubest, off);
      const int orow = __shfl_xor_sync(0xffffffffu, br, off);
      if (ou < ubest || (ou == ubest && orow < br)) {
        ubest = ou;
        br = orow;
      }
    }
    const int bn = a.near[br];
    int bi = min(br, bn), bj = max(br, bn);
    // other pairs whose lower bound reaches it; a stale bound is renewed first
    bool other = bn >= m;  // (no finite distance at all)
#pragma unroll 1
    for (int r0 = 0; r0 < m; r0 += 32) {
      const int r = r0 + lane;
      const bool low2 = r < m && a.lb2[r] <= ubest;
      unsigned stale = __ballot_sync(0xffffffffu, low2 && a.near2[r] == kGone);
#pragma unroll 1
      while (stale != 0u) {
        renew_row(r0 + __ffs(stale) - 1, m);
        stale &= stale - 1u;
      }
      __syncwarp();
      if (r < m) other = other || a.lb2[r] <= ubest || (r != bi && r != bj && a.lb[r] <= ubest);
    }
    double ymin = 0.0;
    if (!__any_sync(0xffffffffu, other)) {
      if (m <= 6) ymin = jet_distance(a, bi, bj, P.inv_s);
    } else {
      if (lane == 0) atomicAdd(&E.counters[5], 1ull);  // merges with several FP64 candidates
      int bp_ = 0x7fffffff;
      ymin = INFINITY;
      bi = 0;
      bj = 1;
      PairWalk w;
      for (w.start(m, lane); w.valid(m); w.next<32>(m)) {
        float u, l;
        pair_bounds(a.f[w.j], a.f[w.k()], u, l);
        if (l > ubest) continue;
        const double yy = jet_distance(a, w.j, w.k(), P.inv_s);
        if (bp_ == 0x7fffffff || yy < ymin) {
          ymin = yy;
          bp_ = w.p;
          bi = w.j;
          bj = w.k();
        }
      }
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const double oy = __shfl_xor_sync(0xffffffffu, ymin, off);
        const int op = __shfl_xor_sync(0xffffffffu, bp_, off), oi = __shfl_xor_sync(0xffffffffu, bi, off);
        const int oj = __shfl_xor_sync(0xffffffffu, bj, off);
        // lanes without a candidate hold position 0x7fffffff
        if (op != 0x7fffffff && (bp_ == 0x7fffffff || oy < ymin || (oy == ymin && op < bp_))) {
          ymin = oy;
          bp_ = op;
          bi = oi;
          bj = oj;
        }
      }
      bi = __shfl_sync(0xffffffffu, bi, 0);  // one pair for all lanes, undefined distances included
      bj = __shfl_sync(0xffffffffu, bj, 0);
    }
    if (m <= 6) yres[m - 3] = ymin;
    if (m == 3) break;
    // jet bi takes the sum, the last jet moves into bj
    const int last = m - 1;
    __syncwarp();  // every lane is done reading the jets of this merge
    if (lane < 4) {
      a.j[lane][bi] += a.j[lane][bj];
      a.j[lane][bj] = a.j[lane][last];
    }
    __syncwarp();
    const float4 moved = a.f[last], merged = direction(bi);
    __syncwarp();
    if (lane == 0) {
      a.f[bj] = moved;  // (bj == last: beyond the jets that are left)
      a.f[bi] = merged;
    }
    __syncwarp();
    // the rows of the jets that are left: those that pointed at the merged
    // ones are renewed, the new jet is offered to the others
#pragma unroll 1
    for (int r0 = 0; r0 < last; r0 += 32) {
      const int r = r0 + lane;
      bool renew = false;
      if (r < last) {
        Row row = load_row(a, r == bj ? last : r);
        renew = r == bi || row.near == bi || row.near == bj;
        if (!renew) {
          if (row.near2 == bi || row.near2 == bj) row.near2 = kGone;
          if (row.near == last) row.near = bj;
          if (row.near2 == last) row.near2 = bj;
          float u, l;
          pair_bounds(a.f[r], merged, u, l);
          row.add(u, l, bi);
          store_row(a, r, row);
        }
      }
      unsigned todo = __ballot_sync(0xffffffffu, renew);
#pragma unroll 1
      while (todo != 0u) {
        renew_row(r0 + __ffs(todo) - 1, last);
        todo &= todo - 1u;
      }
    }
  }
  if (lane == 0)
    for (int h = 0; h < 4; ++h) E.obs[h * E.stride + ev] = yres[h];
}

// ------------------------------------------------------------- buckets
// Parton count of event ev if it gets observables: finished, with 2 ..
// capacity partons (the shower never writes another count; callers that pass
// their own arrays may), else -1.
__device__ __forceinline__ int shape_partons(const Events& E, int64_t ev) {
  if (E.status[ev] != GAPS_DONE) return -1;
  const int n = E.n_partons[ev];
  return n >= 2 && n <= E.cap ? n : -1;
}

// counts[n] = finished events with n partons (2 <= n <= capacity <= 255).
__global__ void __launch_bounds__(256) k_bucket_count(Events E, int* counts, Ranges R) {
  follow_launch();
  __shared__ int sh[256];
  sh[threadIdx.x] = 0;
  __syncthreads();
  for (int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; t < E.n;
       t += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int n = shape_partons(E, R.event(t));
    if (n >= 0) atomicAdd(&sh[n], 1);
  }
  __syncthreads();
  if (sh[threadIdx.x]) atomicAdd(&counts[threadIdx.x], sh[threadIdx.x]);
}

// offsets[n] = first position of bucket n; cursor[n] = offsets[n];
// offsets[256] = number of finished events.
// Clears the observables' counter words too (the kernels behind it count).
__global__ void __launch_bounds__(256) k_bucket_scan(const int* counts, int* offsets, int* cursor,
                                                     unsigned long long* counters) {
  follow_launch();
  __shared__ int sh[256];
  const int t = threadIdx.x;
  if (t == 4 || t == 5 || t == 8) counters[t] = 0ull;
  sh[t] = counts[t];
  __syncthreads();
  for (int d = 1; d < 256; d <<= 1) {
    const int v = t >= d ? sh[t - d] : 0;
    __syncthreads();
    sh[t] += v;
    __syncthreads();
  }
  const int excl = t ? sh[t - 1] : 0;
  offsets[t] = excl;
  cursor[t] = excl;
  if (t == 255) offsets[256] = sh[255];
}

// Finished events go to their bucket; the others get undefined observables,
// and so do finished events with a parton count outside 2 .. capacity
// (counted in counter word 8).
// A warp's lanes of one bucket take their places with one shared-memory
// atomic, a block's with one global atomic per bucket and round, so the
// few hot buckets (a handful of multiplicities hold most events) see a
// thousand times fewer global atomics than with one per event.
__global__ void __launch_bounds__(256) k_bucket_scatter(Events E, int* cursor, int* order, Ranges R) {
  follow_launch();
  __shared__ int s_cnt[256];
  __shared__ int s_base[256];
  const int tid = threadIdx.x, lane = tid & 31;
  for (int64_t first = static_cast<int64_t>(blockIdx.x) * 256; first < E.n;
       first += static_cast<int64_t>(gridDim.x) * 256) {
    s_cnt[tid] = 0;
    __syncthreads();
    const int64_t t = first + tid;
    const int64_t ev = t < E.n ? R.event(t) : 0;
    int n = -1;
    if (t < E.n) {
      n = shape_partons(E, ev);
      if (n < 0) {
        if (E.status[ev] == GAPS_DONE) atomicAdd(&E.counters[8], 1ull);
        for (int h = 0; h < GAPS_N_OBS; ++h) E.obs[h * E.stride + ev] = -1.0;
      }
    }
    const unsigned peers = __match_any_sync(0xffffffffu, n);
    const int leader = __ffs(peers) - 1;
    int at = 0;
    if (n >= 0 && lane == leader) at = atomicAdd(&s_cnt[n], __popc(peers));
    at = __shfl_sync(0xffffffffu, at, leader) + __popc(peers & ((1u << lane) - 1u));
    __syncthreads();
    if (s_cnt[tid]) s_base[tid] = atomicAdd(&cursor[tid], s_cnt[tid]);
    __syncthreads();
    if (n >= 0) order[s_base[n] + at] = static_cast<int>(ev);
    __syncthreads();  // s_cnt and s_base are reused by the next round
  }
}

// Count, scan and scatter of a small batch by one block: the same buckets in
// one launch instead of a clearing and three.
constexpr int64_t kSmallBuckets = 4096;
__global__ void __launch_bounds__(1024) k_buckets_small(Events E, int* offsets, int* cursor, int* order, Ranges R) {
  follow_launch();
  __shared__ int sh[256], place[256];
  const int tid = threadIdx.x;
  constexpr int kEach = static_cast<int>(kSmallBuckets) / 1024;
  int n[kEach];
  int64_t ev[kEach];
  if (tid < 256) sh[tid] = 0;
  if (tid == 4 || tid == 5 || tid == 8) E.counters[tid] = 0ull;
  __syncthreads();
#pragma unroll
  for (int c = 0; c < kEach; ++c) {
    const int64_t t = c * 1024 + tid;
    n[c] = -1;
    if (t >= E.n) continue;
    ev[c] = R.event(t);
    n[c] = shape_partons(E, ev[c]);
    if (n[c] >= 0) {
      atomicAdd(&sh[n[c]], 1);
    } else {
      if (E.status[ev[c]] == GAPS_DONE) atomicAdd(&E.counters[8], 1ull);
      for (int h = 0; h < GAPS_N_OBS; ++h) E.obs[h * E.stride + ev[c]] = -1.0;
    }
  }
  __syncthreads();
  for (int d = 1; d < 256; d <<= 1) {
    const int v = tid < 256 && tid >= d ? sh[tid - d] : 0;
    __syncthreads();
    if (tid < 256) sh[tid] += v;
    __syncthreads();
  }
  if (tid < 256) {
    const int excl = tid ? sh[tid - 1] : 0;
    offsets[tid] = excl;
    place[tid] = excl;
    if (tid == 255) offsets[256] = sh[255];
    if (tid < 2) cursor[tid] = 0;  // the large events' cursors (no event has 0 or 1 partons)
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < kEach; ++c)
    if (n[c] >= 0) order[atomicAdd(&place[n[c]], 1)] = static_cast<int>(ev[c]);
}

// Events of buckets n_lo..n_hi (all with n <= MAXJ), the largest first: the
// order list holds the buckets by rising multiplicity, and the threads take
// it from its end, so the blocks with the costliest events start first and
// the cheap ones fill the SMs that free up (a launch otherwise waits for the
// blocks of its largest events, dealt out last).
template <int MAXJ>
__global__ void __launch_bounds__(kShapeThreads) k_event_shapes(DevParams P, Events E, const int* order,
                                                                const int* offsets, int n_lo, int n_hi) {
  follow_launch();
  const int begin = offsets[n_lo], end = offsets[n_hi + 1 > 256 ? 256 : n_hi + 1];
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < end - begin; j += gridDim.x * blockDim.x) {
    const int64_t ev = order[end - 1 - j];
    event_shapes<MAXJ>(P, E, ev, E.n_partons[ev]);
  }
}

// Events of buckets n_lo..n_hi (all with n <= MAXJ), L lanes per event, T
// threads per block.
template <int MAXJ, int L, int T>
__global__ void __launch_bounds__(T) k_event_shapes_group(DevParams P, Events E, const int* order,
                                                          const int* offsets, int n_lo, int n_hi) {
  follow_launch();
  constexpr int G = T / L;
  __shared__ GroupArrays<MAXJ> s_ev[G];
  const int g = threadIdx.x / L, sub = threadIdx.x % L;
  const unsigned gm = group_lanes<L>();
  const int begin = offsets[n_lo], end = offsets[n_hi + 1 > 256 ? 256 : n_hi + 1];
  for (int k = begin + blockIdx.x * G + g; k < end; k += gridDim.x * G) {
    const int64_t ev = order[k];
    event_shapes_group<MAXJ, L>(P, E, ev, E.n_partons[ev], s_ev[g], sub, gm);
    __syncwarp(gm);  // the group's arrays are free for its next event
  }
}

// Events of buckets n_lo..n_hi (all with n <= MAXJ), a warp each, T threads
// per block, the largest first; the warps of the resident blocks take them
// one by one from *cursor (zero before the launch).
template <int MAXJ, int T, int kBlocks>
__global__ void __launch_bounds__(T, kBlocks) k_event_shapes_warp(DevParams P, Events E, const int* order, const int* offsets,
                                                         int n_lo, int n_hi, int* cursor) {
  follow_launch();
  extern __shared__ __align__(16) unsigned char s_shapes[];
  WarpEvent<MAXJ>& a = reinterpret_cast<WarpEvent<MAXJ>*>(s_shapes)[threadIdx.x >> 5];
  const int lane = static_cast<int>(threadIdx.x & 31);
  const int begin = offsets[n_lo], end = offsets[n_hi + 1 > 256 ? 256 : n_hi + 1];
  if (begin == end) return;
  for (;;) {
    int k = 0;
    if (lane == 0) k = atomicAdd(cursor, 1);
    k = __shfl_sync(0xffffffffu, k, 0);
    if (k >= end - begin) return;
    const int64_t ev = order[end - 1 - k];
    event_shapes_warp<MAXJ>(P, E, ev, E.n_partons[ev], a, lane);
    __syncwarp();  // the arrays are free for the next event
  }
}

// Events of up to 16 partons take one thread each in batches of at least
// kThreadsFrom events (throughput), groups of lanes in smaller ones (a launch
// then waits for its slowest event, not for the SMs), the more the smaller the
// batch: the stage at 10^3 events takes 122, 92 and 72 us with 4, 8 and 16
// lanes, at 2x10^4 138, 122 and 178, at 4.9x10^4 172, 201 and 380; at 10^5 254
// with 4 lanes and 349 with one thread per event, at 3x10^5 613 and 490 us.
// The per-thread grid holds one thread per event up to kShapeBlocksPerSm
// blocks per SM (largest events first, above): 0.86 ms at 10^6 events then; a
// second launch of lane groups for 7, 9, 11 or 13 .. 16 partons there took the
// stage to 1.10, 1.00, 0.99 and 0.93.  All of LEP events (4.9 partons on
// average); the lines take no account of the multiplicities.
constexpr int kShapeBlocksPerSm = 64;
constexpr int64_t kThreadsFrom = 180000;

}  // namespace

cudaError_t preload_observables() {
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, k_bucket_count);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_buckets_small);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_bucket_scan);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_bucket_scatter);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_event_shapes<16>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_event_shapes_group<16, 4, 128>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_event_shapes_group<16, 8, 128>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_event_shapes_group<16, 16, 128>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_event_shapes_warp<128, 128, 5>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_event_shapes_warp<256, 64, 6>);
  return e;
}

cudaError_t launch_observables(const DevParams& P, const Events& E, int* buckets, int* order, cudaStream_t s,
                               const Ranges& R) {
  if (E.n == 0) return cudaSuccess;
  int sms = 152, dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int* counts = buckets;
  int* offsets = buckets + 256;
  int* cursor = buckets + 256 + 257;
  const bool chain = E.n < kChainBelow;
  cudaError_t e = cudaSuccess;
  if (E.n <= kSmallBuckets) {
    e = launch_chained(chain, k_buckets_small, 1, 1024, 0, s, E, offsets, cursor, order, R);
  } else {
    const int64_t want = (E.n + 255) / 256;
    const int64_t grid_count = want < 4 * sms ? want : 4 * sms;
    e = cudaMemsetAsync(counts, 0, 256 * sizeof(int), s);
    if (e == cudaSuccess) e = launch_chained(chain, k_bucket_count, grid_count, 256, 0, s, E, counts, R);
    if (e == cudaSuccess) e = launch_chained(chain, k_bucket_scan, 1, 256, 0, s, counts, offsets, cursor, E.counters);
    if (e == cudaSuccess) e = launch_chained(chain, k_bucket_scatter, grid_count, 256, 0, s, E, cursor, order, R);
  }
  if (e != cudaSuccess) return e;
  // One launch per multiplicity class; grids cover the largest possible
  // class (blocks of one event per thread or per group) and stride over the
  // actual one.
  auto grid = [&](int per_block, int per_sm) {
    const int64_t want = (E.n + per_block - 1) / per_block;
    return static_cast<unsigned>(want < static_cast<int64_t>(per_sm) * sms ? want : static_cast<int64_t>(per_sm) * sms);
  };
  const auto groups = [&](auto lanes) {
    constexpr int L = decltype(lanes)::value;
    return launch_chained(chain, k_event_shapes_group<16, L, 128>, grid(128 / L, 8), 128, 0, s, P, E, order, offsets, 0, 16);
  };
  if (E.n < 10000) {
    e = groups(std::integral_constant<int, 16>{});
  } else if (E.n < 30000) {
    e = groups(std::integral_constant<int, 8>{});
  } else if (E.n < kThreadsFrom) {
    e = groups(std::integral_constant<int, 4>{});
  } else {
    e = launch_chained(chain, k_event_shapes<16>, grid(kShapeThreads, kShapeBlocksPerSm), kShapeThreads, 0, s, P, E, order,
                       offsets, 0, 16);
  }
  // One class up to 128 partons (96 registers leave five blocks per SM), one
  // beyond.  Their cursors are the bucket cursors of 0 and 1 partons, which no
  // event has: zero.
  if (e == cudaSuccess && E.cap > 16)
    e = launch_chained(chain, k_event_shapes_warp<128, 128, 5>, grid(4, 5), 128, 4 * sizeof(WarpEvent<128>), s, P, E, order,
                       offsets, 17, 128, cursor);
  if (e == cudaSuccess && E.cap > 128)
    e = launch_chained(chain, k_event_shapes_warp<256, 64, 6>, grid(2, 6), 64, 2 * sizeof(WarpEvent<256>), s, P, E, order,
                       offsets, 129, 255, cursor + 1);
  return e;
}

}  // namespace gaps

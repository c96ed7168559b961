// The Ls-direction operator on the lanes of a site: a thread holds the 24 reals of
// two adjacent slices, the Ls/2 threads of a site are consecutive lanes of one warp.
#pragma once

#include "device_common.cuh"

namespace dwf {

// Lanes of one site: the np = Ls/2 thread pairs of a site are consecutive lanes
// of one warp (sites never straddle a warp), so slice s0 - 1 is the second
// slice of lane - 1 (of lane + np - 1 for s0 = 0) and slice s0 + 2 the first
// slice of lane + 1 (of lane - np + 1 for the last pair).
struct PairLanes {
  int up, dn;       // source lanes of slices s0 - 1 and s0 + 2
  float fm, fp;     // their wrap factors (-m_f across the Ls boundary, else 1)
};
__device__ __forceinline__ PairLanes pair_lanes(int lane, int jp, int np, float mf) {
  PairLanes pl;
  pl.up = jp == 0 ? lane + np - 1 : lane - 1;
  pl.dn = jp == np - 1 ? lane - (np - 1) : lane + 1;
  pl.fm = jp == 0 ? -mf : 1.f;
  pl.fp = jp == np - 1 ? -mf : 1.f;
  return pl;
}

// One chirality of ls_lanes with the inverse, 12 reals of the slices 2 jp (a0) and
// 2 jp + 1 (a1): z = (p0 + p1 S) y, y = (1 - r S)^-1 v, on the lanes of the site as a
// scan (no shared memory). DOWN: S takes s - 1. There the wrap-free recursion yh_j =
// v_j + r yh_{j-1} (yh_0 = v_0) is a scan over the site's lanes with the constant factor
// r^2 per lane (C: yh at the lane's second slice); the wrap then adds r^j d with d =
// -m_f r yh_{Ls-1} / (1 + m_f r^Ls) (the closed form's first element). Where S takes
// s + 1 the same runs in reversed order. One step of the scan runs over all 12
// components, which share its factors. The scan only gives y at the place before
// the lane's first slice; the lane's own y follow from it by the recursion, one
// rounding each, as when a thread walks the column: every step of the scan rounds C
// again, and y taken from there had an error 13 % larger. REFINE: the recursion once
// more, from the neighbour's y, for kernels that have the time (M_5^-1 waits for HBM); it
// takes what is left of the scan's error out (Shamir, Ls = 32: 3 %). The larger term, p0,
// is the one that is not rounded before the sum.
template <bool DOWN, bool REFINE>
__device__ __forceinline__ void ls_half_inverse(float *a0, float *a1, int Ls, int np, int jp, int lane,
                                                const LsK<float> &c, const PairLanes &pl) {
  const float r = c.r, p0 = c.p0q, p1 = c.p1q, mfr = -c.mf * c.r * c.inv_den;
  const int j = DOWN ? jp : np - 1 - jp;  // the lane's place in the order
  const int src = DOWN ? pl.up : pl.dn, end = lane - jp + (DOWN ? np - 1 : 0);
  const float wrap = DOWN ? pl.fm : pl.fp, rw = r * wrap, pw = p1 * wrap;
  // r^(2 j - 1) at the place before the lane's first slice (the wrap: r^(Ls - 1))
  const int e = j > 0 ? 2 * j - 1 : Ls - 1;
  float g = 1.f;
  for (int i = 0; i < e; ++i) g *= r;
  float *first = DOWN ? a0 : a1, *second = DOWN ? a1 : a0;
  float C[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) C[k] = fmaf(r, first[k], second[k]);
  float m = r * r;
  for (int d = 1; d < np; d <<= 1) {
    // (selected, not multiplied by zero: the lane d away may be another site's)
    const bool on = j >= d;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const float t = DOWN ? __shfl_up_sync(0xffffffffu, C[k], d) : __shfl_down_sync(0xffffffffu, C[k], d);
      if (on) C[k] = fmaf(m, t, C[k]);
    }
    m *= m;
  }
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const float last = __shfl_sync(0xffffffffu, C[k], end), cin = __shfl_sync(0xffffffffu, C[k], src);
    float before = fmaf(g, mfr * last, cin);
    if constexpr (REFINE)
      before = __shfl_sync(0xffffffffu, fmaf(r, fmaf(rw, before, first[k]), second[k]), src);
    const float yf = fmaf(rw, before, first[k]), ys = fmaf(r, yf, second[k]);
    first[k] = fmaf(p0, yf, pw * before);
    second[k] = fmaf(p0, ys, p1 * yf);
  }
}

// (a0, a1) <- q0 (p0 + p1 S) [(1 - r S)^-1] (a0, a1), the slices 2 jp and 2 jp + 1.
// Every lane of the warp calls this; only lanes of the same site are used.
template <bool DAG, bool REFINE = false>
__device__ __forceinline__ void ls_lanes(float (&a0)[24], float (&a1)[24], bool inv, int Ls, int np,
                                         int jp, int lane, const LsK<float> &c,
                                         const PairLanes &pl) {
  const float p0 = c.p0q, p1 = c.p1q;
  if (inv) {
    ls_half_inverse<!DAG, REFINE>(a0, a1, Ls, np, jp, lane, c, pl);
    ls_half_inverse<DAG, REFINE>(a0 + 12, a1 + 12, Ls, np, jp, lane, c, pl);
  } else if (p1 != 0.f) {
    // q0 (p0 + p1 S) needs only the neighbouring slices: the pair's own and
    // the outer ones from the neighbouring lanes of the site
#pragma unroll
    for (int k = 0; k < 24; ++k) {
      const bool down = (k < 12) != DAG;  // S takes s - 1 on these components
      const float wu = __shfl_sync(0xffffffffu, a1[k], pl.up);
      const float wd = __shfl_sync(0xffffffffu, a0[k], pl.dn);
      const float t0 = a0[k], t1 = a1[k];
      if (down) {
        a0[k] = fmaf(p0, t0, p1 * (pl.fm * wu));
        a1[k] = fmaf(p0, t1, p1 * t0);
      } else {
        a0[k] = fmaf(p0, t0, p1 * t1);
        a1[k] = fmaf(p0, t1, p1 * (pl.fp * wd));
      }
    }
  } else {
#pragma unroll
    for (int k = 0; k < 24; ++k) {
      a0[k] *= p0;
      a1[k] *= p0;
    }
  }
}

}  // namespace dwf

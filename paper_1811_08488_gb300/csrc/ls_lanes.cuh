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

// (a0, a1) <- q0 (p0 + p1 S) [(1 - r S)^-1] (a0, a1), the slices 2 jp and 2 jp + 1.
// Every lane of the warp calls this; only lanes of the same site are used.
template <bool DAG>
__device__ __forceinline__ void ls_lanes(float (&a0)[24], float (&a1)[24], bool inv, int Ls, int np,
                                         int jp, int lane, const LsK<float> &c,
                                         const PairLanes &pl) {
  const float p0 = c.p0q, p1 = c.p1q;
  if (inv) {
    // z = (p0 + p1 S) y, y = (1 - r S)^-1 v, on the lanes of the site as a scan (no
    // shared memory). On the components where S takes s - 1: the wrap-free
    // recursion yh_j = v_j + r yh_{j-1} (yh_0 = v_0) is a scan over the
    // site's lanes with the constant factor r^2 per lane (C: yh at the lane's
    // second slice); the wrap then adds r^j d with d = -m_f r yh_{Ls-1} / (1 + m_f
    // r^Ls) (the closed form's first element). Where S takes s + 1 the same runs
    // in reversed order. One step of the scan runs over all 24 components, which
    // share its factors; y at the neighbour that p1 S needs follows from the
    // lane's own copy of C there.
    const float r = c.r, mfr = -c.mf * c.r * c.inv_den;
    const int base = lane - jp, jr = np - 1 - jp;  // the lane's place in either order
    float rd = 1.f, ru = 1.f, rl = 1.f;            // r^(2 jp), r^(2 jr), r^(Ls - 1)
    for (int i = 0; i < 2 * jp; ++i) rd *= r;
    for (int i = 0; i < 2 * jr; ++i) ru *= r;
    for (int i = 0; i < Ls - 1; ++i) rl *= r;
    float C[24];
#pragma unroll
    for (int k = 0; k < 24; ++k) {
      const bool down = (k < 12) != DAG;
      C[k] = down ? fmaf(r, a0[k], a1[k]) : fmaf(r, a1[k], a0[k]);
    }
    float m = r * r;
    for (int d = 1; d < np; d <<= 1) {
      // (selected, not multiplied by zero: the lane d away may be another site's)
      const bool od = jp >= d, ou = jr >= d;
#pragma unroll
      for (int k = 0; k < 24; ++k) {
        const bool down = (k < 12) != DAG;
        const float t = down ? __shfl_up_sync(0xffffffffu, C[k], d)
                             : __shfl_down_sync(0xffffffffu, C[k], d);
        if (down ? od : ou) C[k] = fmaf(m, t, C[k]);
      }
      m *= m;
    }
    // r^(2 j - 1) at the place before the lane's first slice (the wrap: r^(Ls - 1))
    float gd = rl, gu = rl;
    if (jp > 0) {
      gd = r;
      for (int i = 0; i < 2 * jp - 2; ++i) gd *= r;
    }
    if (jr > 0) {
      gu = r;
      for (int i = 0; i < 2 * jr - 2; ++i) gu *= r;
    }
    const float pd = p1 * pl.fm, pu = p1 * pl.fp;
#pragma unroll
    for (int k = 0; k < 24; ++k) {
      const bool down = (k < 12) != DAG;
      const float cin = down ? __shfl_up_sync(0xffffffffu, C[k], 1)
                             : __shfl_down_sync(0xffffffffu, C[k], 1);
      const float last = __shfl_sync(0xffffffffu, C[k], down ? base + np - 1 : base);
      const float dl = mfr * last;
      const float first = down ? a0[k] : a1[k];  // v at the first slice of the order
      const float rf = down ? rd : ru;
      const bool inner = (down ? jp : jr) > 0;
      const float yf = fmaf(rf, dl, fmaf(r, inner ? cin : 0.f, first));
      const float ys = fmaf(rf * r, dl, C[k]);
      const float before = fmaf(down ? gd : gu, dl, inner ? cin : last);
      const float zf = fmaf(down ? pd : pu, before, p0 * yf);
      const float zs = fmaf(p1, yf, p0 * ys);
      a0[k] = down ? zf : zs;
      a1[k] = down ? zs : zf;
    }
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
        a0[k] = p0 * t0 + p1 * (pl.fm * wu);
        a1[k] = p0 * t1 + p1 * t0;
      } else {
        a0[k] = p0 * t0 + p1 * t1;
        a1[k] = p0 * t1 + p1 * (pl.fp * wd);
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

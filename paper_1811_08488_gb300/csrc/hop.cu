// The 4D Wilson hop with the fifth dimension, the one kernel behind every
// operator application of the solver (paper Sec. 2.2, M^4 = D^w M_phi and
// eq. for D^w; Sec. 2.3 for its use inside the Dirichlet block operator).
//
// Two kernels. hop2_kernel (FP32/FP16/BF16 fields, even Ls): one thread per
// pair of slices (s0, s0 + 1) of one output site; the Ls/2 threads of a site
// are consecutive lanes of one warp (a warp holds whole sites), and everything
// that couples neighbouring slices -- M_phi on load (s0 - 1, s0 + 2), the Ls
// epilogue (M_phi^+, M_5^-1, K = M_phi M_5^-1 and their adjoints) and the x-term
// of the epilogue -- is exchanged between those lanes with warp shuffles; the
// epilogue's (1 - r S)^-1 is a scan over the site's lanes.
//
// What bounds hop2_kernel: 16 warps per SM (48 accumulators a thread) waiting for
// the gather, 8 x 96 bytes per element in FP32 through L2 (gather and stores alone:
// 318 us on 24^3 x 64 x 16, FP32 adjoint). Two things shorten the wait:
// - The links are staged in shared memory once per CTA. Read by every lane of a
//   site they were 5 of the 11 loads of a direction for 1/20 of its bytes, and
//   without them the adjoint hop took 353 us instead of 513.
// - The next direction's spinors are loaded into the registers that the projection
//   has just freed, while the projected spins are multiplied by the link.
// And the Ls epilogue's scan runs one step over all 24 components at a time, with
// shared factors, 480 instead of about 1100 instructions per thread.
// Measured on 24^3 x 64 x 16, before -> now: FP32 M^4 613 -> 504 us, adjoint
// 513 -> 397, FP16 642 -> 483 and 433 -> 373. Not kept:
// rings of stages in shared memory filled by cp.async or by TMA boxes, all
// bit-identical: the work to issue them (150 instructions a direction beside 230 of
// arithmetic) and the larger code cost more than the waiting they save (853 and
// 883 us for FP32 M^4); mma.m16n8k16 for FP16 fields (one site per warp: 968
// instructions per site instead of 553, 660 us for the adjoint); an L2 prefetch
// of the rows that come next (FP32 M^4 631 us, adjoint 535).
//
// The other form of the kernel (DENSE = false) runs direction by direction, leaves out
// those that no lane has, and reads the links where they are: for the outer ring of a
// block's region, whose sites have one or two neighbours, and where staging does not
// pay (hop_staged_sites has the rule and its measurements).
//
// hop_kernel (FP64 fields, odd Ls): one thread per output (site, s), the Ls
// epilogue walks columns in shared memory.
//
// For output site x and direction mu (chiral basis, g_mu = [[0, A],[A^+, 0]]):
//   forward : (1 - sg g_mu) U_mu(x)      chi(x+mu)
//   backward: (1 + sg g_mu) U_mu(x-mu)^+ chi(x-mu)
// with sg = +1 for Dhop and sg = -1 for Dhop^+. (1 - g)v = [h; -A^+ h] with
// h = v_u - A v_l, so only the two-spinor h is multiplied by the link.
// With PRE, the input is chi = M_phi psi = b psi + c C psi, formed on load:
// chi_u(s) = b psi_u(s) + c psi_u(s-1), chi_l(s) = b psi_l(s) + c psi_l(s+1),
// with the wrap factor -m_f.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "device_common.cuh"
#include "ls_lanes.cuh"

namespace dwf {

template <class R>
struct Cx {
  R re, im;
};

// (A v_l) for the two lower spins v2, v3 -> a0, a1 (per colour).
template <int MU, class R>
__device__ __forceinline__ void a_times(const Cx<R> v2, const Cx<R> v3, Cx<R> &a0, Cx<R> &a1) {
  if constexpr (MU == 0) {  // A = -i sigma_1
    a0 = {v3.im, -v3.re};
    a1 = {v2.im, -v2.re};
  } else if constexpr (MU == 1) {  // A = -i sigma_2 = [[0,-1],[1,0]]
    a0 = {-v3.re, -v3.im};
    a1 = {v2.re, v2.im};
  } else if constexpr (MU == 2) {  // A = -i sigma_3 = diag(-i, i)
    a0 = {v2.im, -v2.re};
    a1 = {-v3.im, v3.re};
  } else {  // A = 1
    a0 = v2;
    a1 = v3;
  }
}

// (A^+ w) for the two projected spins w0, w1 -> b0, b1.
template <int MU, class R>
__device__ __forceinline__ void adag_times(const Cx<R> w0, const Cx<R> w1, Cx<R> &b0, Cx<R> &b1) {
  if constexpr (MU == 0) {  // A^+ = i sigma_1
    b0 = {-w1.im, w1.re};
    b1 = {-w0.im, w0.re};
  } else if constexpr (MU == 1) {  // A^+ = [[0,1],[-1,0]]
    b0 = w1;
    b1 = {-w0.re, -w0.im};
  } else if constexpr (MU == 2) {  // A^+ = diag(i, -i)
    b0 = {-w0.im, w0.re};
    b1 = {w1.im, -w1.re};
  } else {
    b0 = w0;
    b1 = w1;
  }
}

template <class R, int MU, bool FWD, bool DAG, bool PAIRS>
__device__ __forceinline__ void proj_mul_acc(R *acc, const R *v, const R *u);

// One direction of the hop: project, multiply by U or U^+, reconstruct, add.
// `lk` is the link record.
template <class S, int MU, bool FWD, bool DAG, bool PRE, bool RC, bool PAIRS>
__device__ __forceinline__ void hop_dir(typename S::R *acc, const char *in, long long soff,
                                        int cs, int j, int s, int Ls, const uint4 *lk,
                                        size_t ls, const LsCoef &cf) {
  using R = typename S::R;
  R v[24];
  load24<S>(in, soff, cs, j * Ls + s, v);
  if constexpr (PRE) {
    R w[12];
    const LsK<R> &kk = kc<R>(cf);
    const R b = kk.pre_b, c = kk.pre_c, mf = kk.mf;
    const int sm = s == 0 ? Ls - 1 : s - 1;
    const R fm = s == 0 ? -mf : (R)1;
    load12<S, true>(in, soff, cs, j * Ls + sm, w);
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = fma(b, v[k], c * fm * w[k]);
    const int sp = s == Ls - 1 ? 0 : s + 1;
    const R fp = s == Ls - 1 ? -mf : (R)1;
    load12<S, false>(in, soff, cs, j * Ls + sp, w);
#pragma unroll
    for (int k = 0; k < 12; ++k) v[12 + k] = fma(b, v[12 + k], c * fp * w[k]);
  }
  R u[18];
  load_link<S>(lk, ls, u, RC ? 1 : 0);
  proj_mul_acc<R, MU, FWD, DAG, PAIRS>(acc, v, u);
}

// Project v with (1 - sg g_mu), multiply the two-spinor by U (forward) or U^+
// (backward), reconstruct and add to acc. In FP64 the FP64 pipe is the bound
// (a DFMA takes 65 cycles per warp and scheduler), so U h is a chain of 72
// multiply-adds: `re += ur * hr - ui * hi` compiles to a product, a
// multiply-add and a sum, 108 operations. Measured with M_phi taken out of D_PC's hops
// (mphi_input) and whole warps (hop_sites_per_cta): A in FP64 on
// 16^3 x 32 x 12 8.57 -> 5.59 ms, 0.69 of the FP64 pipe's rate. Its error, against 80-bit
// arithmetic, is 0.94 to 0.98 of what it was for D_PC and A. A single hop has nothing to
// make up for the chain's 1 to 2 %: its products are summed in pairs (PAIRS).
// FP32 and FP16 (odd Ls) wait for their gather and take what has no larger error than
// before: pairs with M_phi on load, the sums of Re U h and Im U h apart otherwise. As
// one chain the error of one hop is 4 to 6 % larger.
template <class R, int MU, bool FWD, bool DAG, bool PAIRS>
__device__ __forceinline__ void proj_mul_acc(R *acc, const R *v, const R *u) {
  constexpr bool kChain = std::is_same<R, double>::value && !PAIRS;
  constexpr R sg = (FWD != DAG) ? (R)1 : (R)-1;  // projector (1 - sg g_mu)
  Cx<R> h[2][3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    Cx<R> v0{v[0 * 6 + 2 * c], v[0 * 6 + 2 * c + 1]};
    Cx<R> v1{v[1 * 6 + 2 * c], v[1 * 6 + 2 * c + 1]};
    Cx<R> v2{v[2 * 6 + 2 * c], v[2 * 6 + 2 * c + 1]};
    Cx<R> v3{v[3 * 6 + 2 * c], v[3 * 6 + 2 * c + 1]};
    Cx<R> a0, a1;
    a_times<MU>(v2, v3, a0, a1);
    h[0][c] = {v0.re - sg * a0.re, v0.im - sg * a0.im};
    h[1][c] = {v1.re - sg * a1.re, v1.im - sg * a1.im};
  }
  Cx<R> w[2][3];
#pragma unroll
  for (int sp = 0; sp < 2; ++sp) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      R re, im, re2, im2;  // (the products with Re U and with Im U)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        // forward: U[a][b]; backward: conj(U[b][a])
        const R ur = FWD ? u[2 * (3 * a + b)] : u[2 * (3 * b + a)];
        const R ui = FWD ? u[2 * (3 * a + b) + 1] : -u[2 * (3 * b + a) + 1];
        const R hr = h[sp][b].re, hi = h[sp][b].im;
        if constexpr (kChain) {
          re = b == 0 ? ur * hr : fma(ur, hr, re);
          re = fma(-ui, hi, re);
          im = b == 0 ? ur * hi : fma(ur, hi, im);
          im = fma(ui, hr, im);
        } else if constexpr (PAIRS) {
          const R pr = fma(ur, hr, -ui * hi), pi = fma(ur, hi, ui * hr);
          re = b == 0 ? pr : re + pr;
          im = b == 0 ? pi : im + pi;
        } else {
          re = b == 0 ? ur * hr : fma(ur, hr, re);
          re2 = b == 0 ? ui * hi : fma(ui, hi, re2);
          im = b == 0 ? ur * hi : fma(ur, hi, im);
          im2 = b == 0 ? ui * hr : fma(ui, hr, im2);
        }
      }
      if constexpr (!kChain && !PAIRS) {
        re -= re2;
        im += im2;
      }
      w[sp][a] = {re, im};
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    Cx<R> b0, b1;
    adag_times<MU>(w[0][c], w[1][c], b0, b1);
    acc[0 * 6 + 2 * c] += w[0][c].re;
    acc[0 * 6 + 2 * c + 1] += w[0][c].im;
    acc[1 * 6 + 2 * c] += w[1][c].re;
    acc[1 * 6 + 2 * c + 1] += w[1][c].im;
    acc[2 * 6 + 2 * c] -= sg * b0.re;
    acc[2 * 6 + 2 * c + 1] -= sg * b0.im;
    acc[3 * 6 + 2 * c] -= sg * b1.re;
    acc[3 * 6 + 2 * c + 1] -= sg * b1.im;
  }
}

template <class S, int MU, bool DAG, bool PRE, bool RC, bool PAIRS>
__device__ __forceinline__ void hop_mu(typename S::R *acc, const HopParams &P, const char *in,
                                       const uint4 *links, const int *nb, int site, int s,
                                       const LsCoef &cf) {
  constexpr int LC = RC ? S::kLinkChunksRecon : S::kLinkChunks;
  const int jf = nb[2 * MU], jb = nb[2 * MU + 1];
  const size_t ls = (size_t)P.link_cs;
  const uint4 *lmu = links + (size_t)MU * LC * ls;
  if (jf >= 0 && jf < P.in_limit)
    hop_dir<S, MU, true, DAG, PRE, RC, PAIRS>(acc, in, P.in.scale_off, P.in.cs, jf, s, P.Ls,
                                   lmu + P.out_link_off + site, ls, cf);
  if (jb >= 0 && jb < P.in_limit)
    hop_dir<S, MU, false, DAG, PRE, RC, PAIRS>(acc, in, P.in.scale_off, P.in.cs, jb, s, P.Ls,
                                    lmu + P.in_link_off + jb, ls, cf);
}

// Shared memory of one CTA for the Ls epilogue: the hop result T and the
// own-site input X as [site][component][Ls + 1] columns.
template <class R>
__device__ __forceinline__ void epilogue_columns(R *T, const R *X, int nsites, int site0,
                                                 int n_out, int Ls, bool dag, int inv,
                                                 const LsCoef &cf) {
  const int col = Ls + 1;
  for (int w = threadIdx.x; w < nsites * 24; w += blockDim.x) {
    if (site0 + w / 24 >= n_out) continue;
    const bool down = ((w % 24) < 12) != dag;
    ls_column<R>(T + w * col, X ? X + w * col : nullptr, Ls, down, inv != 0, kc<R>(cf));
  }
}

// One thread's part of the fused <dotv, out> of the global dot products. The
// FP32 products are summed with Kahan compensation, so the sum's error is at
// most about 3 * 2^-24 * sum |d_k a_k| (one rounding per product, two for the
// compensated sum) whatever the count; the partials are then added in FP64.
// FP64 fields sum in FP64.
template <class R>
__device__ __forceinline__ double dot_compensated(const R *d, const R *a, int n) {
  if constexpr (std::is_same<R, double>::value) {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 24; ++k)
      if (k < n) s += d[k] * a[k];
    return s;
  } else {
    float s = 0.f, c = 0.f;
#pragma unroll
    for (int k = 0; k < 24; ++k)
      if (k < n) {
        const float y = d[k] * a[k] - c;
        const float t = s + y;
        c = (t - s) - y;
        s = t;
      }
    return (double)s - (double)c;
  }
}

// Publish the CTA's part of Re<dotv, out> (both summed per (rhs, block)).
__device__ __forceinline__ void hop_dot(const HopParams &P, double d, double *red, int rhs,
                                        int blk) {
  d = cta_sum(d, red);
  const int ntiles = gridDim.x;
  const int grp = rhs * P.nblocks + blk;
  double total;
  if (group_reduce(d, P.partials + (size_t)grp * ntiles, ntiles, blockIdx.x, P.counters + grp,
                   total))
    P.dot_out[(size_t)rhs * P.dot_rstride + blk] = total;
}

// Kernel timer (only when P.prof is set). CTA 0 reads the global timer at
// entry (CTAs are dispatched in index order, so it starts first); every CTA
// takes a ticket when it has finished, and the CTA with the last ticket reads
// the timer again, adds the span to the slot and resets it for the next
// launch. One atomic per CTA. Launches of one slot must not overlap in time
// (one stream at a time), which stream order guarantees.
__device__ __forceinline__ unsigned long long gtimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ bool first_cta() {
  return blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0;
}
__device__ __noinline__ void prof_enter(const HopParams &P) {
  if (P.prof && threadIdx.x == 0 && first_cta()) {
    P.prof->start = gtimer_ns();
    __threadfence();
  }
}
__device__ __noinline__ void prof_exit(const HopParams &P) {
  if (!P.prof) return;
  __syncthreads();
  if (threadIdx.x != 0) return;
  KernProf *k = P.prof;
  const unsigned int nct = gridDim.x * gridDim.y * gridDim.z;
  if (atomicAdd(&k->done, 1u) != nct - 1) return;
  __threadfence();
  const unsigned long long t1 = gtimer_ns();
  const unsigned long long t0 = *reinterpret_cast<volatile unsigned long long *>(&k->start);
  k->total_ns += t1 - t0;
  if (!P.prof_again) k->launches += 1;
  k->bytes += P.alg_bytes;
  k->done = 0;
  __threadfence();
}

// One thread per output (site, s): used for FP64 fields and odd Ls. PAIRS: how U h is summed
// (proj_mul_acc).
template <class S, bool DAG, bool PRE, bool RC, bool PAIRS>
__device__ __forceinline__ void hop_body(const HopParams &P) {
  using R = typename S::R;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  const int rhs = blockIdx.z, blk = blockIdx.y;
  if (P.skip && P.skip[rhs]) return;
  if (P.bskip && P.bskip[rhs * P.nblocks + blk]) return;
  const int Ls = P.Ls;
  const int nsites = P.nsites;  // blockDim.x is nsites * Ls rounded up to whole warps
  const int tid = threadIdx.x;
  const int s = tid % Ls, sl = tid / Ls;
  const int site0 = blockIdx.x * nsites;
  const int site = site0 + sl;
  const bool active = (sl < nsites) && (site < P.n_out);
  const LsCoef &cf = P.coef[rhs];

  const char *in = P.in.data + blk * P.in.bstride + rhs * P.in.rstride;
  char *out = P.out.data + blk * P.out.bstride + rhs * P.out.rstride;
  const uint4 *links = reinterpret_cast<const uint4 *>(P.links + blk * P.link_bstride);

  R acc[24];
#pragma unroll
  for (int k = 0; k < 24; ++k) acc[k] = 0;
  if (active) {
    const int *nb = P.nbr + (size_t)site * 8;
    hop_mu<S, 0, DAG, PRE, RC, PAIRS>(acc, P, in, links, nb, site, s, cf);
    hop_mu<S, 1, DAG, PRE, RC, PAIRS>(acc, P, in, links, nb, site, s, cf);
    hop_mu<S, 2, DAG, PRE, RC, PAIRS>(acc, P, in, links, nb, site, s, cf);
    hop_mu<S, 3, DAG, PRE, RC, PAIRS>(acc, P, in, links, nb, site, s, cf);
  }
  const int e = site * Ls + s;

  if (P.epi) {
    const int col = Ls + 1;
    R *T = reinterpret_cast<R *>(smem_raw);
    R *X = T + nsites * 24 * col;
    if (active) {
#pragma unroll
      for (int k = 0; k < 24; ++k) T[(sl * 24 + k) * col + s] = acc[k];
      if (P.has_x) {
        R xv[24];
        if (site < P.xown_limit) {
          const char *xo = P.xown.data + blk * P.xown.bstride + rhs * P.xown.rstride;
          load24<S>(xo, P.xown.scale_off, P.xown.cs, e, xv);
        } else {
#pragma unroll
          for (int k = 0; k < 24; ++k) xv[k] = 0;
        }
#pragma unroll
        for (int k = 0; k < 24; ++k) X[(sl * 24 + k) * col + s] = xv[k];
      }
    }
    __syncthreads();
    epilogue_columns<R>(T, P.has_x ? X : nullptr, nsites, site0, P.n_out, Ls, DAG, P.inv, cf);
    __syncthreads();
    if (active) {
#pragma unroll
      for (int k = 0; k < 24; ++k) acc[k] = T[(sl * 24 + k) * col + s];
    }
  } else {
    const R q = kc<R>(cf).q0;
#pragma unroll
    for (int k = 0; k < 24; ++k) acc[k] *= q;
  }
  if (active) store24<S>(out, P.out.scale_off, P.out.cs, e, acc);

  if (P.dot) {
    double d = 0.0;
    if (active) {
      R dv[24];
      const char *dp = P.dotv.data + blk * P.dotv.bstride + rhs * P.dotv.rstride;
      load24<S>(dp, P.dotv.scale_off, P.dotv.cs, e, dv);
      d = dot_compensated<R>(dv, acc, 24);
    }
    hop_dot(P, d, red, rhs, blk);
  }
}

// CTAs per SM: FP32 with M_phi on load has too many values for three (80 registers: it
// spilled, and took 84.9 us instead of 70.9 on 16^3 x 32, Ls = 7; with 128 registers 66.7),
// the others gain from the third (adjoint 96.8 -> 78.0 us). FP64 CTAs have at most 128
// threads and their registers are left to the compiler.
template <class S, bool DAG, bool PRE, bool RC>
__global__ void __launch_bounds__(256, std::is_same<S, F32>::value &&PRE ? 2 : 3)
    hop_kernel(const __grid_constant__ HopParams P) {
  prof_enter(P);
  hop_body<S, DAG, PRE, RC, PRE>(P);
  prof_exit(P);
}
template <bool DAG, bool PRE, bool PAIRS>
__global__ void __launch_bounds__(256) hop64_kernel(const __grid_constant__ HopParams P) {
  prof_enter(P);
  hop_body<F64, DAG, PRE, false, PAIRS>(P);
  prof_exit(P);
}
// single: the hop is the whole operator (FP64: summed in pairs, see proj_mul_acc)
template <class S, bool DAG, bool PRE, bool RC>
static auto hop_entry(bool single) {
  if constexpr (std::is_same<S, F64>::value)
    return PRE || single ? hop64_kernel<DAG, PRE, true> : hop64_kernel<DAG, PRE, PRE>;
  else
    return hop_kernel<S, DAG, PRE, RC>;
}

constexpr int kHopCtas = 4;  // CTAs of hop2_kernel per SM (128 registers a thread)

// ---------------------------------------------------------------------------
// Two slices per thread: thread (site, s0 = 2j) computes s0 and s0 + 1. Chunk c
// of both slices is one 32-byte word, so every spinor load and store is a
// 256-bit access and a warp moves one contiguous kilobyte per instruction; the
// link serves both slices; with M_phi on load, the two slices
// supply each other's s -> s +- 1 neighbours and only the outer two halves
// (s0 - 1 upper, s0 + 2 lower) are loaded in addition. Arithmetic runs on
// float2 pairs (slice s0, slice s0 + 1) with Blackwell's packed FP32
// instructions, so each multiply-add serves both slices. FP32/FP16/BF16, even Ls.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 bc(float a) { return make_float2(a, a); }
// x + sgn * y on both lanes (sgn = +-1 at compile time): one packed FMA.
template <int SGN>
__device__ __forceinline__ float2 pm(float2 x, float2 y) {
  return __ffma2_rn(y, make_float2((float)SGN, (float)SGN), x);
}
struct C2 {
  float2 re, im;
};
// x + sgn * (ph * z), ph = i^PH (PH = 0: 1, 1: i, 2: -1, 3: -i).
template <int PH, int SGN>
__device__ __forceinline__ C2 add_phase(C2 x, C2 z) {
  if constexpr (PH == 0) return {pm<SGN>(x.re, z.re), pm<SGN>(x.im, z.im)};
  else if constexpr (PH == 1) return {pm<-SGN>(x.re, z.im), pm<SGN>(x.im, z.re)};
  else if constexpr (PH == 2) return {pm<-SGN>(x.re, z.re), pm<-SGN>(x.im, z.im)};
  else return {pm<SGN>(x.re, z.im), pm<-SGN>(x.im, z.re)};
}
// (A v_l)_sp = i^PH v_l[SRC]: per direction mu, for output spin 0 and 1.
template <int MU> struct ProjA;
template <> struct ProjA<0> { static constexpr int s0 = 1, p0 = 3, s1 = 0, p1 = 3; };  // -i s1
template <> struct ProjA<1> { static constexpr int s0 = 1, p0 = 2, s1 = 0, p1 = 0; };  // -i s2
template <> struct ProjA<2> { static constexpr int s0 = 0, p0 = 3, s1 = 1, p1 = 1; };  // -i s3
template <> struct ProjA<3> { static constexpr int s0 = 0, p0 = 0, s1 = 1, p1 = 0; };  // 1
// (A^+ w)_sp = i^PH w[SRC].
template <int MU> struct ProjAd;
template <> struct ProjAd<0> { static constexpr int s0 = 1, p0 = 1, s1 = 0, p1 = 1; };
template <> struct ProjAd<1> { static constexpr int s0 = 1, p0 = 0, s1 = 0, p1 = 2; };
template <> struct ProjAd<2> { static constexpr int s0 = 0, p0 = 1, s1 = 1, p1 = 3; };
template <> struct ProjAd<3> { static constexpr int s0 = 0, p0 = 0, s1 = 1, p1 = 0; };

// x + y * s on both lanes (s = the two slices' scales, or their negatives).
__device__ __forceinline__ float2 fma_s(float2 x, float2 y, float2 s) { return __ffma2_rn(y, s, x); }
// x + sgn * sc * (ph * z): add_phase with the slices' scales folded in.
template <int PH, int SGN>
__device__ __forceinline__ C2 add_phase_s(C2 x, C2 z, float2 sp, float2 sn) {
  const float2 a = SGN > 0 ? sp : sn, b = SGN > 0 ? sn : sp;  // +sgn*sc, -sgn*sc
  if constexpr (PH == 0) return {fma_s(x.re, z.re, a), fma_s(x.im, z.im, a)};
  else if constexpr (PH == 1) return {fma_s(x.re, z.im, b), fma_s(x.im, z.re, a)};
  else if constexpr (PH == 2) return {fma_s(x.re, z.re, b), fma_s(x.im, z.im, b)};
  else return {fma_s(x.re, z.im, a), fma_s(x.im, z.re, b)};
}

// Packed counterpart of proj_mul_acc in two parts; v, h and acc hold both slices.
// h = (1 - SG g_mu) v, the two projected spins.
struct HalfSpinor {
  C2 h[2][3];
};
template <int MU, bool FWD, bool DAG>
__device__ __forceinline__ void project2(HalfSpinor &p, const float2 *v) {
  constexpr int SG = (FWD != DAG) ? 1 : -1;  // projector (1 - SG g_mu)
  using A = ProjA<MU>;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const C2 vu0{v[0 * 6 + 2 * c], v[0 * 6 + 2 * c + 1]};
    const C2 vu1{v[1 * 6 + 2 * c], v[1 * 6 + 2 * c + 1]};
    const C2 vl[2] = {{v[2 * 6 + 2 * c], v[2 * 6 + 2 * c + 1]},
                      {v[3 * 6 + 2 * c], v[3 * 6 + 2 * c + 1]}};
    p.h[0][c] = add_phase<A::p0, -SG>(vu0, vl[A::s0]);
    p.h[1][c] = add_phase<A::p1, -SG>(vu1, vl[A::s1]);
  }
}
// acc += the spinor reconstructed from U h (U^+ h backward). SCALED: h came from
// stored FP16/BF16 values whose per-slice scales sc are applied in the
// accumulation (the projector and U are linear).
template <int MU, bool FWD, bool DAG, bool SCALED = false>
__device__ __forceinline__ void mul_acc2(float2 *acc, const HalfSpinor &p, const float *u,
                                         float2 sc = make_float2(1.f, 1.f)) {
  constexpr int SG = (FWD != DAG) ? 1 : -1;
  using Ad = ProjAd<MU>;
  const float2 scn = make_float2(-sc.x, -sc.y);
  C2 w[2][3];
#pragma unroll
  for (int sp = 0; sp < 2; ++sp) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      float2 re = make_float2(0.f, 0.f), im = make_float2(0.f, 0.f);
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        // forward: U[a][b]; backward: conj(U[b][a])
        const float ur = FWD ? u[2 * (3 * a + b)] : u[2 * (3 * b + a)];
        const float ui = FWD ? u[2 * (3 * a + b) + 1] : -u[2 * (3 * b + a) + 1];
        re = __ffma2_rn(bc(ur), p.h[sp][b].re, re);
        re = __ffma2_rn(bc(-ui), p.h[sp][b].im, re);
        im = __ffma2_rn(bc(ur), p.h[sp][b].im, im);
        im = __ffma2_rn(bc(ui), p.h[sp][b].re, im);
      }
      w[sp][a] = {re, im};
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if constexpr (SCALED) {
      acc[0 * 6 + 2 * c] = fma_s(acc[0 * 6 + 2 * c], w[0][c].re, sc);
      acc[0 * 6 + 2 * c + 1] = fma_s(acc[0 * 6 + 2 * c + 1], w[0][c].im, sc);
      acc[1 * 6 + 2 * c] = fma_s(acc[1 * 6 + 2 * c], w[1][c].re, sc);
      acc[1 * 6 + 2 * c + 1] = fma_s(acc[1 * 6 + 2 * c + 1], w[1][c].im, sc);
    } else {
      acc[0 * 6 + 2 * c] = __fadd2_rn(acc[0 * 6 + 2 * c], w[0][c].re);
      acc[0 * 6 + 2 * c + 1] = __fadd2_rn(acc[0 * 6 + 2 * c + 1], w[0][c].im);
      acc[1 * 6 + 2 * c] = __fadd2_rn(acc[1 * 6 + 2 * c], w[1][c].re);
      acc[1 * 6 + 2 * c + 1] = __fadd2_rn(acc[1 * 6 + 2 * c + 1], w[1][c].im);
    }
    const C2 l0{acc[2 * 6 + 2 * c], acc[2 * 6 + 2 * c + 1]};
    const C2 l1{acc[3 * 6 + 2 * c], acc[3 * 6 + 2 * c + 1]};
    C2 n0, n1;
    if constexpr (SCALED) {
      n0 = add_phase_s<Ad::p0, -SG>(l0, w[Ad::s0][c], sc, scn);
      n1 = add_phase_s<Ad::p1, -SG>(l1, w[Ad::s1][c], sc, scn);
    } else {
      n0 = add_phase<Ad::p0, -SG>(l0, w[Ad::s0][c]);
      n1 = add_phase<Ad::p1, -SG>(l1, w[Ad::s1][c]);
    }
    acc[2 * 6 + 2 * c] = n0.re;
    acc[2 * 6 + 2 * c + 1] = n0.im;
    acc[3 * 6 + 2 * c] = n1.re;
    acc[3 * 6 + 2 * c + 1] = n1.im;
  }
}

// ---------------------------------------------------------------------------
// Links in shared memory. The Ls/2 lanes of a site all need its 8 links; read from
// global memory by each lane they cost as many L1 requests as the spinors for a
// twentieth of the bytes. The CTA copies the links of its sites once, 16
// bytes per lane, to [direction][word][site] and every lane reads them from there.
// ---------------------------------------------------------------------------
template <class S, bool RC> __host__ __device__ constexpr int link_words() {
  return RC ? S::kLinkChunksRecon : S::kLinkChunks;
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}
// Start the copy (128 threads). An absent neighbour's link is zero. FP16 records are widened to the FP32 record on the way, once per link instead of by
// each of the site's lanes (conversions run on the FMA pipe, 8 x 18 of them per
// lane otherwise).
template <class S, bool RC>
__device__ __forceinline__ void stage_links(uint4 *sl, const HopParams &P, const uint4 *links,
                                            int site0) {
  constexpr int LC = link_words<S, RC>(), LS = link_words<F32, RC>();
  const size_t ls = (size_t)P.link_cs;
  for (int e = threadIdx.x; e < 8 * P.nsites; e += 128) {
    const int d = e / P.nsites, i = e - d * P.nsites, site = site0 + i;
    if (site >= P.n_out) continue;
    const uint4 *lmu = links + (size_t)(d >> 1) * LC * ls;
    uint4 *dst = sl + d * LS * P.nsites;
    const int j = __ldg(P.nbr + (size_t)site * 8 + d);
    if ((unsigned)j >= (unsigned)P.in_limit) {
#pragma unroll
      for (int w = 0; w < LS; ++w) dst[w * P.nsites + i] = make_uint4(0u, 0u, 0u, 0u);
      continue;
    }
    const uint4 *src = lmu + ((d & 1) ? P.in_link_off + j : P.out_link_off + site);
    if constexpr (S::kHalf) {
      float t[8 * LC];
#pragma unroll
      for (int w = 0; w < LC; ++w) unpack8<F16>(__ldg(src + w * ls), t + 8 * w);
#pragma unroll
      for (int w = 0; w < LS; ++w)
        dst[w * P.nsites + i] = make_uint4(__float_as_uint(t[4 * w]), __float_as_uint(t[4 * w + 1]),
                                           __float_as_uint(t[4 * w + 2]), __float_as_uint(t[4 * w + 3]));
    } else {
#pragma unroll
      for (int w = 0; w < LC; ++w) cp_async16(dst + w * P.nsites + i, src + w * ls);
    }
  }
  if constexpr (!S::kHalf) asm volatile("cp.async.commit_group;" ::: "memory");
}
template <class S>
__device__ __forceinline__ void wait_links() {
  if constexpr (!S::kHalf) asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
}

// The input of one direction as loaded (FP16/BF16 without their scales).
struct DirIn {
  float v0[24], v1[24];
  float2 sc;
};
template <class S>
__device__ __forceinline__ void load_dir2(DirIn &in2, const char *in, long long soff, int cs,
                                          int e) {
  if constexpr (S::kHalf)
    load24x2_unscaled<S>(in, soff, cs, e, in2.v0, in2.v1, in2.sc);
  else
    load24x2<S>(in, soff, cs, e, in2.v0, in2.v1);
}

__device__ __forceinline__ void zero_dir2(DirIn &d) {
#pragma unroll
  for (int k = 0; k < 24; ++k) d.v0[k] = d.v1[k] = 0.f;
  d.sc = make_float2(0.f, 0.f);
}

// The projected spins of one direction from its loaded input.
template <class S, int MU, bool FWD, bool DAG, bool PRE>
__device__ __forceinline__ void dir_project(HalfSpinor &h, const DirIn &d, const LsCoef &cf,
                                            const PairLanes &pl) {
  float2 v[24];
  if constexpr (PRE) {
    // M_phi on both slices as packed FMAs: (chi(s0), chi(s0+1)) =
    // b (v(s0), v(s0+1)) + c (shifted neighbours); the outer halves come
    // from the neighbouring lanes of the same site (all lanes take part). FP16/BF16: the
    // wrap factors and the slices' scales are folded into the coefficients. FP32: the
    // wrap factor is applied to the outer half; folded in, the coefficients are pairs of
    // their own in every lane, and M^4 without staged links took 1 to 2 % longer.
    const float b = cf.f.pre_b, c = cf.f.pre_c;
    float2 bs = bc(b), cu = bc(c), cl = bc(c);
    if constexpr (S::kHalf) {
      const float sm = __shfl_sync(0xffffffffu, d.sc.y, pl.up);
      const float sp = __shfl_sync(0xffffffffu, d.sc.x, pl.dn);
      bs = make_float2(b * d.sc.x, b * d.sc.y);
      cu = make_float2(c * pl.fm * sm, c * d.sc.x);
      cl = make_float2(c * d.sc.y, c * pl.fp * sp);
    }
    const float fm = S::kHalf ? 1.f : pl.fm, fp = S::kHalf ? 1.f : pl.fp;
#pragma unroll
    for (int k = 0; k < 12; ++k) {  // upper: chi(s0) <- s0-1, chi(s0+1) <- s0
      const float w = __shfl_sync(0xffffffffu, d.v1[k], pl.up);
      v[k] = __ffma2_rn(cu, make_float2(fm * w, d.v0[k]),
                        __fmul2_rn(bs, make_float2(d.v0[k], d.v1[k])));
    }
#pragma unroll
    for (int k = 12; k < 24; ++k) {  // lower: chi(s0) <- s0+1, chi(s0+1) <- s0+2
      const float w = __shfl_sync(0xffffffffu, d.v0[k], pl.dn);
      v[k] = __ffma2_rn(cl, make_float2(d.v1[k], fp * w),
                        __fmul2_rn(bs, make_float2(d.v0[k], d.v1[k])));
    }
  } else {
#pragma unroll
    for (int k = 0; k < 24; ++k) v[k] = make_float2(d.v0[k], d.v1[k]);
  }
  project2<MU, FWD, DAG>(h, v);
}
// Its contribution; lk: the site's link (STAGED: in shared memory), words ls apart.
template <class S, int MU, bool FWD, bool DAG, bool PRE, bool RC, bool STAGED>
__device__ __forceinline__ void dir_add(float2 *acc, const HalfSpinor &h, float2 sc, const uint4 *lk,
                                        size_t ls) {
  constexpr bool kFold = !PRE && S::kHalf;  // scales folded into the FMAs
  float u[18];
  if constexpr (STAGED)
    load_link<F32, true>(lk, ls, u, RC ? 1 : 0);
  else
    load_link<S>(lk, ls, u, RC ? 1 : 0);
  mul_acc2<MU, FWD, DAG, kFold>(acc, h, u, kFold ? sc : make_float2(1.f, 1.f));
}

// The x-term of the Ls epilogue, out += (a0 + a1 S) x, on the thread's slices
// s0 and s0 + 1 (o0, o1), added after the column walk. S is the walk's chiral
// shift: (S x)_s = x_{s-1} with (S x)_0 = -mf x_{Ls-1} on the components the
// walk runs down (the upper spin components of the operator, the lower ones
// of its adjoint), (S x)_s = x_{s+1} with (S x)_{Ls-1} = -mf x_0 on the
// others. Besides the pair it needs the down half of x at s0 - 1 and the up
// half at s0 + 2.
// Every lane of the warp calls this (the halves of slices s0 - 1 and s0 + 2
// come from the neighbouring lanes); `have` is false where x is zero.
template <class S, bool DAG>
__device__ __forceinline__ void add_x_term2(float *o0, float *o1, const char *x, long long soff,
                                            int cs, int site, int s0, int Ls, bool have,
                                            const LsK<float> &c, const PairLanes &pl) {
  float x0[12], x1[12], w[12];
  const int e = site * Ls + s0;
  const float a0 = c.a0, a1 = c.a1;
  const float fm = pl.fm, fp = pl.fp;
  // upper components: down for the operator, up for its adjoint
  if (have) {
    load12x2<S, true>(x, soff, cs, e, x0, x1);
  } else {
#pragma unroll
    for (int k = 0; k < 12; ++k) x0[k] = x1[k] = 0.f;
  }
#pragma unroll
  for (int k = 0; k < 12; ++k)
    w[k] = DAG ? __shfl_sync(0xffffffffu, x0[k], pl.dn) : __shfl_sync(0xffffffffu, x1[k], pl.up);
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    if (!DAG) {
      o0[k] += a0 * x0[k] + a1 * (fm * w[k]);
      o1[k] += a0 * x1[k] + a1 * x0[k];
    } else {
      o0[k] += a0 * x0[k] + a1 * x1[k];
      o1[k] += a0 * x1[k] + a1 * (fp * w[k]);
    }
  }
  // lower components: up for the operator, down for its adjoint
  if (have) {
    load12x2<S, false>(x, soff, cs, e, x0, x1);
  } else {
#pragma unroll
    for (int k = 0; k < 12; ++k) x0[k] = x1[k] = 0.f;
  }
#pragma unroll
  for (int k = 0; k < 12; ++k)
    w[k] = DAG ? __shfl_sync(0xffffffffu, x1[k], pl.up) : __shfl_sync(0xffffffffu, x0[k], pl.dn);
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    if (!DAG) {
      o0[12 + k] += a0 * x0[k] + a1 * x1[k];
      o1[12 + k] += a0 * x1[k] + a1 * (fp * w[k]);
    } else {
      o0[12 + k] += a0 * x0[k] + a1 * (fm * w[k]);
      o1[12 + k] += a0 * x1[k] + a1 * x0[k];
    }
  }
}

// EPI: the Ls epilogue is compiled in (its column registers would otherwise
// weigh on the plain hop's register allocation).
template <class S, bool DAG, bool PRE, bool RC, bool EPI, bool DENSE>
__device__ __forceinline__ void hop2_body(const HopParams &P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  const int rhs = blockIdx.z, blk = blockIdx.y;
  if (P.skip && P.skip[rhs]) return;
  if (P.bskip && P.bskip[rhs * P.nblocks + blk]) return;
  const int Ls = P.Ls, np = Ls >> 1;
  const int nsites = P.nsites;  // (blockDim.x / 32) * (32 / np): whole sites per warp
  const int tid = threadIdx.x, lane = tid & 31, spw = 32 / np;
  const int jp = lane % np, slw = lane / np;
  const int sl = (tid >> 5) * spw + slw;
  const int s0 = 2 * jp;
  const int site0 = P.site_off + blockIdx.x * nsites;
  const int site = site0 + sl;
  const bool active = (slw < spw) && (site < P.n_out);
  const LsCoef &cf = P.coef[rhs];
  const PairLanes pl = pair_lanes(lane, jp, np, cf.f.mf);

  const char *in = P.in.data + blk * P.in.bstride + rhs * P.in.rstride;
  char *out = P.out.data + blk * P.out.bstride + rhs * P.out.rstride;
  const uint4 *links = reinterpret_cast<const uint4 *>(P.links + blk * P.link_bstride);

  float2 acc[24];
#pragma unroll
  for (int k = 0; k < 24; ++k) acc[k] = make_float2(0.f, 0.f);
  DirIn d;
#define HOP_LOAD(J) load_dir2<S>(d, in, P.in.scale_off, P.in.cs, (J) * Ls + s0)
#define HOP_PROJECT(D) \
  HalfSpinor h;        \
  dir_project<S, (D) / 2, ((D) & 1) == 0, DAG, PRE>(h, d, cf, pl);
  if constexpr (DENSE) {
    // Every direction runs; where a neighbour is absent the link is zero (and
    // nbr_read names another neighbour of the site). The next direction's spinors
    // are loaded while this one's projected spins are multiplied (not for FP32
    // with M_phi on load, whose registers that would spill); the links arrive while
    // the first spinors are on their way.
    constexpr bool kPipe = S::kHalf || !PRE;
    constexpr int LC = link_words<F32, RC>();
    // Lanes without a site read what the last site of their warp (the last site of
    // all) reads, which costs nothing more. When they read the neighbours of site 0, lines
    // that every warp of the chip asked for at once, the FP32 adjoint hop on 16^3 x 32 took
    // 63.6 instead of 59.6 us with Ls = 12 and 73.9 instead of 64.0 with Ls = 14.
    const int site_r = min(site0 + (tid >> 5) * spw + min(slw, spw - 1), P.n_out - 1);
    const int *nb = P.nbr_read + (size_t)site_r * 8;
    uint4 *sl_links = reinterpret_cast<uint4 *>(smem_raw);
    stage_links<S, RC>(sl_links, P, links, site0);
    const uint4 *lk = sl_links + (site_r - site0);
#define HOP_DIR(D, NEXT)                                                                      \
  {                                                                                           \
    if (!kPipe && (D) > 0) HOP_LOAD(__ldg(nb + (D)));                                         \
    HOP_PROJECT(D)                                                                            \
    const float2 sc = d.sc;                                                                   \
    if (kPipe) { NEXT; }                                                                      \
    dir_add<S, (D) / 2, ((D) & 1) == 0, DAG, PRE, RC, true>(acc, h, sc, lk + (D) * LC * nsites, \
                                                            nsites);                          \
  }
    HOP_LOAD(__ldg(nb));
    wait_links<S>();
    if constexpr (kPipe) {
      HOP_DIR(0, HOP_LOAD(__ldg(nb + 1)))
      HOP_DIR(1, HOP_LOAD(__ldg(nb + 2)))
      HOP_DIR(2, HOP_LOAD(__ldg(nb + 3)))
      HOP_DIR(3, HOP_LOAD(__ldg(nb + 4)))
      HOP_DIR(4, HOP_LOAD(__ldg(nb + 5)))
      HOP_DIR(5, HOP_LOAD(__ldg(nb + 6)))
      HOP_DIR(6, HOP_LOAD(__ldg(nb + 7)))
      HOP_DIR(7, )
    } else {
      // always taken: keeps the compiler from mixing the directions (and spilling)
      if (P.dirs & 1) HOP_DIR(0, )
      if (P.dirs & 2) HOP_DIR(1, )
      if (P.dirs & 4) HOP_DIR(2, )
      if (P.dirs & 8) HOP_DIR(3, )
      if (P.dirs & 16) HOP_DIR(4, )
      if (P.dirs & 32) HOP_DIR(5, )
      if (P.dirs & 64) HOP_DIR(6, )
      if (P.dirs & 128) HOP_DIR(7, )
    }
#undef HOP_DIR
  } else {
    // With M_phi on load every lane of the warp takes part in a direction (its
    // halves are exchanged between lanes) and one that no lane has is skipped by
    // all; otherwise each lane branches on its own neighbour. A lane without the
    // neighbour loads nothing.
    constexpr int LC = link_words<S, RC>();
    const size_t ls = (size_t)P.link_cs;
    const int4 *nb = reinterpret_cast<const int4 *>(P.nbr + (size_t)(active ? site : 0) * 8);
    const int4 lo = __ldg(nb), hi = __ldg(nb + 1);
    const int js[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#define HOP_DIR(D)                                                                             \
  {                                                                                            \
    const int j = active ? js[D] : -1;                                                         \
    const bool valid = (unsigned)j < (unsigned)P.in_limit;                                     \
    if (PRE ? __any_sync(0xffffffffu, valid) != 0 : valid) {                                   \
      if (!PRE || valid)                                                                       \
        HOP_LOAD(j);                                                                           \
      else                                                                                     \
        zero_dir2(d);                                                                          \
      HOP_PROJECT(D)                                                                           \
      if (valid)                                                                               \
        dir_add<S, (D) / 2, ((D) & 1) == 0, DAG, PRE, RC, false>(                              \
            acc, h, d.sc,                                                                      \
            links + (size_t)((D) / 2) * LC * ls +                                              \
                (((D) & 1) ? P.in_link_off + j : P.out_link_off + site),                       \
            ls);                                                                               \
    }                                                                                          \
  }
    HOP_DIR(0)
    HOP_DIR(1)
    HOP_DIR(2)
    HOP_DIR(3)
    HOP_DIR(4)
    HOP_DIR(5)
    HOP_DIR(6)
    HOP_DIR(7)
#undef HOP_DIR
  }
#undef HOP_PROJECT
#undef HOP_LOAD
  const int e = site * Ls + s0;
  float a0[24], a1[24];
#pragma unroll
  for (int k = 0; k < 24; ++k) {
    a0[k] = acc[k].x;
    a1[k] = acc[k].y;
  }

  if constexpr (EPI) {
    ls_lanes<DAG>(a0, a1, P.inv != 0, Ls, np, jp, lane, cf.f, pl);
    // the x-term, (a0 + a1 S) x, after the Ls operator, in registers; every
    // lane takes part in the exchange of the outer halves
    if (P.has_x) {
      const char *xo = P.xown.data + blk * P.xown.bstride + rhs * P.xown.rstride;
      add_x_term2<S, DAG>(a0, a1, xo, P.xown.scale_off, P.xown.cs, active ? site : 0, s0, Ls,
                          active && site < P.xown_limit, cf.f, pl);
    }
  } else {
    const float q = cf.f.q0;
#pragma unroll
    for (int k = 0; k < 24; ++k) {
      a0[k] *= q;
      a1[k] *= q;
    }
  }
  if (active) store24x2<S>(out, P.out.scale_off, P.out.cs, e, a0, a1);

  if (P.dot) {
    double d = 0.0;
    if (active) {
      float d0[24], d1[24];
      const char *dp = P.dotv.data + blk * P.dotv.bstride + rhs * P.dotv.rstride;
      load24x2<S>(dp, P.dotv.scale_off, P.dotv.cs, e, d0, d1);
      d = dot_compensated<float>(d0, a0, 24) + dot_compensated<float>(d1, a1, 24);
    }
    hop_dot(P, d, red, rhs, blk);
  }
}

template <class S, bool DAG, bool PRE, bool RC, bool EPI, bool DENSE>
__global__ void __launch_bounds__(128, kHopCtas) hop2_kernel(const __grid_constant__ HopParams P) {
  prof_enter(P);
  hop2_body<S, DAG, PRE, RC, EPI, DENSE>(P);
  prof_exit(P);
}

int sm_count() {
  constexpr int kDevices = 64;
  static std::atomic<int> cache[kDevices];  // 0 until read
  int dev = 0, n = 0;
  DWF_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < kDevices && (n = cache[dev].load(std::memory_order_relaxed)) > 0) return n;
  DWF_CUDA_TRY(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev));
  if (dev < kDevices) cache[dev].store(n, std::memory_order_relaxed);
  return n;
}

// Two slices per thread for FP32/FP16/BF16 with even Ls; one otherwise.
static bool hop_pairs(int Ls, dwf_prec p) { return p != DWF_FP64 && Ls % 2 == 0; }

// Sites per CTA. The one-slice kernel takes as many as its largest CTA holds; in FP64,
// between a half and a whole of that, the number that leaves the fewest idle lanes in the
// last warp: a warp instruction of the FP64 pipe takes as long with idle lanes (Ls =
// 12: 8 sites fill three warps, 10 sites leave 8 of 128 lanes idle). For the other types,
// which wait for the gather, that made more CTAs for nothing (12 x 10 x 14 x 18, Ls = 7,
// FP16 adjoint: 22.7 against 18.7 us).
int hop_sites_per_cta(int Ls, dwf_prec p) {
  if (hop_pairs(Ls, p)) return 4 * (32 / (Ls / 2));  // four warps of whole sites
  const int most = (p == DWF_FP64 ? 128 : 256) / Ls;
  if (p != DWF_FP64) return most;
  int best = most;
  auto lanes = [&](int n) { return (n * Ls + 31) / 32 * 32; };
  for (int n = most; n >= 1 && 2 * n >= most; --n)
    if (n * lanes(best) > best * lanes(n)) best = n;
  // (a few per cent at least: three warps are shared worse between the four schedulers
  // than four; 12 x 10 x 14 x 18, Ls = 6, M^4 with 16 sites instead of 21 316 against 281 us)
  return 100 * best * lanes(most) >= 103 * most * lanes(best) ? best : most;
}

// How many leading output sites of a hop (0, n_out, or whole CTAs of the n_dense that
// have all or most neighbours) run with staged links, the others direction by direction;
// fields: blocks x right-hand sides. Measured with against without staged links, 1 wave =
// 4 CTAs on every SM:
// - A staged link serves the Ls/2 lanes of a site. With one lane the copy takes 82 KB of
//   the SM's shared memory and two CTAs fit, with two lanes it saves little (24^3 x 48, FP16
//   adjoint: 112 against 53 us with Ls = 2, 100 against 91 with Ls = 4).
// - All sites, FP16/BF16: with M_phi on load it pays from two lanes on at every size (24^3 x
//   48: 117 against 127 us with Ls = 4, 364 against 467 with Ls = 16), the hops without it
//   from four lanes on (Ls = 8: 158 against 168, Ls = 6: 140 against 138).
// - All sites, FP32: below two waves the wait for the links before the first direction
//   shows (16^4, Ls = 6, 1.35 waves: 22.8 against 20.7 us, adjoint 19.3 against 16.7;
//   16^3 x 32, 2.7 waves: 43.2 against 47.0 and 37.3 against 38.3), but not from six lanes
//   on, with M_phi on load twelve (12^3 x 16, Ls = 24: 34.2 against 37.1, adjoint 26.9
//   against 28.9).
// - Some sites, then a second launch (about 2 us, and a last wave of its own) for the rest;
//   k = 3 preconditioner, FP16 hop 1 (M_phi on load): two launches gain 1 % from 3 waves
//   (8^3 x 16 blocks of 16^3 x 32, Ls = 8: 3.4 waves), lose 1 to 3 % below (2.7 and 1.4).
//   FP32 hop 2: gains 1 to 2 % from 24 waves (12^3 x 16 blocks, Ls = 10), loses 1 to 2 % at 6
//   to 10. FP16 hop 2 and FP32 hop 1: no gain at any size.
int hop_staged_sites(int Ls, dwf_prec p, int dagger, int pre, int n_dense, int n_out,
                     long long fields, int sms) {
  if (!hop_pairs(Ls, p) || n_dense <= 0) return 0;
  const int lanes = Ls / 2, nsites = hop_sites_per_cta(Ls, p);
  const int ctas = (std::min(n_dense, n_out) + nsites - 1) / nsites;
  const int nd = std::min(n_out, ctas * nsites);
  const bool half = p != DWF_FP32;
  int fewest, waves;  // lanes of a site and waves of CTAs that it takes
  if (nd < n_out) {
    if (dagger || half != (pre != 0)) return 0;
    fewest = 3;
    waves = half ? 3 : 24;
  } else if (half) {
    fewest = pre ? 2 : 4;
    waves = 0;
  } else {
    fewest = 3;
    waves = lanes >= (pre ? 12 : 6) ? 0 : 2;
  }
  return lanes >= fewest && ctas * fields >= (long long)waves * kHopCtas * sms ? nd : 0;
}

size_t hop_smem_bytes(int Ls, dwf_prec p, int epi, int has_x, int recon) {
  // the two-slice kernel keeps the 8 links of its sites there
  if (hop_pairs(Ls, p))
    return (size_t)hop_sites_per_cta(Ls, p) * 8 * link_record_bytes(DWF_FP32, recon);
  if (!epi) return 0;
  // the one-slice kernel walks the columns of T (and of x) in shared memory
  const size_t rs = (p == DWF_FP64) ? 8 : 4;
  return (size_t)hop_sites_per_cta(Ls, p) * 24 * (Ls + 1) * rs * (has_x ? 2 : 1);
}

template <class S, bool DAG, bool PRE, bool RC, bool DENSE>
static void launch_two(const HopParams &P, dim3 grid, size_t smem, cudaStream_t st) {
  if (P.epi) {
    hop2_kernel<S, DAG, PRE, RC, true, DENSE><<<grid, 128, smem, st>>>(P);
  } else {
    if constexpr (DAG)
      throw Error{DWF_ERR_UNSUPPORTED, "the adjoint hop always has its M_phi^+ epilogue"};
    else
      hop2_kernel<S, DAG, PRE, RC, false, DENSE><<<grid, 128, smem, st>>>(P);
  }
  DWF_CUDA_TRY(cudaGetLastError());
}

template <class S, bool DAG, bool PRE, bool RC>
static void launch_t(const HopParams &P0, int nrhs, cudaStream_t st, dwf_prec prec) {
  HopParams P = P0;
  for (int r = 0; r < nrhs; ++r) finalize_coef(P.coef[r]);
  const int nsites = hop_sites_per_cta(P.Ls, prec);
  P.nsites = nsites;
  dim3 grid((P.n_out + nsites - 1) / nsites, P.nblocks, nrhs);
  const size_t smem = hop_smem_bytes(P.Ls, prec, P.epi, P.has_x, RC ? 1 : 0);
  if (grid.x == 0) return;
  if constexpr (!std::is_same<S, F64>::value) {
    if (hop_pairs(P.Ls, prec)) {
      // the sites with staged links (whole CTAs of them), then the others
      const int n_out = P.n_out;
      const int nd = hop_staged_sites(P.Ls, prec, DAG, PRE, P.n_dense, n_out,
                                      (long long)P.nblocks * nrhs, sm_count());
      if (nd > 0) {
        P.n_out = nd;
        grid.x = (nd + nsites - 1) / nsites;
        launch_two<S, DAG, PRE, RC, true>(P, grid, smem, st);
      }
      if (nd < n_out) {
        DWF_REQUIRE(nd == 0 || !P.dot, DWF_ERR_UNSUPPORTED, "a fused dot takes one launch");
        P.n_out = n_out;
        P.site_off = nd;
        P.prof_again = nd > 0 ? 1 : 0;
        if (nd > 0) P.alg_bytes = 0;
        grid.x = (n_out - nd + nsites - 1) / nsites;
        launch_two<S, DAG, PRE, RC, false>(P, grid, 0, st);
      }
      return;
    }
  }
  dim3 block((nsites * P.Ls + 31) / 32 * 32);
  hop_entry<S, DAG, PRE, RC>(!P.inv && !P.has_x)<<<grid, block, smem, st>>>(P);
  DWF_CUDA_TRY(cudaGetLastError());
}

template <class S> static dwf_prec prec_of();
template <> dwf_prec prec_of<F64>() { return DWF_FP64; }
template <> dwf_prec prec_of<F32>() { return DWF_FP32; }
template <> dwf_prec prec_of<F16>() { return DWF_FP16; }
template <> dwf_prec prec_of<BF16>() { return DWF_BF16; }

template <class S>
void launch_hop(const HopParams &P, int dagger, int pre_mphi, int nrhs, cudaStream_t st) {
  DWF_REQUIRE(!(dagger && pre_mphi), DWF_ERR_UNSUPPORTED, "M_phi on load is for Dhop only");
  const dwf_prec p = prec_of<S>();
  if constexpr (!std::is_same<S, F64>::value) {
    if (P.recon) {
      if (dagger)
        launch_t<S, true, false, true>(P, nrhs, st, p);
      else if (pre_mphi)
        launch_t<S, false, true, true>(P, nrhs, st, p);
      else
        launch_t<S, false, false, true>(P, nrhs, st, p);
      return;
    }
  }
  DWF_REQUIRE(!P.recon, DWF_ERR_UNSUPPORTED, "FP64 links are never reconstructed");
  if (dagger)
    launch_t<S, true, false, false>(P, nrhs, st, p);
  else if (pre_mphi)
    launch_t<S, false, true, false>(P, nrhs, st, p);
  else
    launch_t<S, false, false, false>(P, nrhs, st, p);
}

// Allow the one-slice hop kernels more than 48 KB of dynamic shared memory (staged links
// take 41 KB at most). Called once per device before any launch (and so before any
// stream capture).
template <class K>
static void allow_big_smem(K *kernel) {
  DWF_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    200 * 1024));
}
template <class S>
static void prepare_one() {
  for (bool single : {false, true}) {
    allow_big_smem(hop_entry<S, false, false, false>(single));
    allow_big_smem(hop_entry<S, false, true, false>(single));
    allow_big_smem(hop_entry<S, true, false, false>(single));
    if constexpr (!std::is_same<S, F64>::value) {
      allow_big_smem(hop_entry<S, false, false, true>(single));
      allow_big_smem(hop_entry<S, false, true, true>(single));
      allow_big_smem(hop_entry<S, true, false, true>(single));
    }
  }
}
void prepare_kernels() {
  prepare_one<F64>();
  prepare_one<F32>();
  prepare_one<F16>();
  prepare_one<BF16>();
}

template void launch_hop<F64>(const HopParams &, int, int, int, cudaStream_t);
template void launch_hop<F32>(const HopParams &, int, int, int, cudaStream_t);
template void launch_hop<F16>(const HopParams &, int, int, int, cudaStream_t);
template void launch_hop<BF16>(const HopParams &, int, int, int, cudaStream_t);

}  // namespace dwf

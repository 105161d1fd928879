// Truncation SVD of a two-qubit gate: pivoted Gram-Schmidt, then one-sided
// Jacobi sweeps (Algorithm 1 of the paper's "SVD and one-side jacobi"
// subsection) on the triangular factor, and the truncation.
//
// A = C~ is m x n (m = 2 chi_l rows, n = 2 chi_r columns, A[r, c] =
// lam_q[r / 2] C[r, c]).  Modified Gram-Schmidt with column pivoting gives A =
// Q R (only R is kept; R is as accurate as a Householder factorisation's), and
// the sweeps orthogonalise the columns of X = R^H (n x r, r the numerical
// rank): X J = W Sigma.  W's columns are the right singular vectors of A (Q
// drops out), so the rows of B~_{q+1} are the conjugated, normalised columns
// of X J, and nothing accumulates V.  Drmac and Veselic (SIAM J. Matrix Anal.
// Appl. 29, 2008, "New fast and accurate Jacobi SVD algorithm") give the
// reason for the factorisation: the columns of X are graded and, scaled to
// unit norm, well conditioned, so the sweeps converge in 4 to 11 instead of 15
// to 60, every column keeps its relative accuracy (normalising small columns
// is safe, unlike columns of A itself), and the columns are n long instead of
// the m + n of [A; V].  r is often about half of n: a theta B_q B_{q+1} has
// rank at most chi_m times the gate's Schmidt rank.
//
// Work split.  One CTA while the columns are few (no barrier between SMs),
// else a cluster of P CTAs, or a grid of P co-resident CTAs for thetas whose
// columns do not fit a cluster's shared memory.  X is split into 2P blocks;
// CTA p holds the blocks at positions p and 2P-1-p of a circle-method round
// robin, each round pairs the columns of its two blocks (in the first round
// also inside each block), then the blocks advance one position.  Blocks move
// through a global workspace that stays in L2 (each CTA writes its blocks to
// their home place, one barrier, each reads its new ones): half the shared
// memory of a ping-pong hand-over, and the same code for cluster and grid.
//
// What it measured (one theta, against FP32-then-double-float sweeps of [A; V]
// on 8 CTAs, which it replaced): 124 x 124 over ten decades 19.5 -> 4.4 ms (36
// -> 10 sweeps), 62 x 94 of rank 31 8.2 -> 0.89 ms, 512 x 512 1.20 s -> 47 ms
// (8 CTAs -> a grid of 128), 16 x 16 in FP64 1.10 -> 0.57 ms.  It is bound by
// the dependent pair steps, one block barrier each (at 124 x 124 the FP32 pipe is
// busy for 37 % of the time; most stalls are at that barrier, where the 8 of 16
// warps that have no pair wait; the cluster barrier comes 7 times a sweep).
//
// A pair of columns is one step of a group of 8 to 32 lanes: as few lanes as
// give every warp a pair, because the angle and the reductions cost each
// group the same.  Norms are kept and updated (|x'|^2 = |x|^2 - t|g|); a
// Gram entry is one complex dot product.  In double-float, sweeps that still
// find large couplings take it from the FP32 heads.
#pragma once

#include <cooperative_groups.h>

#include <cstring>
#include <type_traits>

#include "common.cuh"
#include "svd_arith.cuh"

namespace mpsv {

namespace cg = cooperative_groups;

// The theta is scaled by a power of two to a largest entry near 2^40: squares
// of columns 17 decades smaller, and the error terms of those squares, then
// stay far from the ends of the FP32 range.  Columns below 1e-17 of the largest
// entry (less than FP64 rounding) count as zero.
constexpr int kScaleExp = 40;
constexpr float kZeroNorm2 = 1e-34f * 1.2089258e24f;  // (1e-17 2^40)^2

// ---- teams: the CTAs that work on one theta --------------------------------
// publish / candidate exchange one (value, index) pair per CTA in each
// Gram-Schmidt step; remote() reads another CTA's column.  barrier() returns,
// for the whole CTA alike, whether every CTA arrived: where it is false (only a
// grid can give up) what the others published must not be read, and the CTA
// leaves at once.

struct OneTeam {
  static constexpr bool kGlobalA = false;
  static constexpr int me = 0, P = 1;
  __device__ bool barrier() {
    __syncthreads();
    return true;
  }
};

struct ClusterTeam {
  static constexpr bool kGlobalA = false;
  int me, P;
  float2* mail;  // shared memory: [2][16] candidates
  int barriers = 0;
  __device__ bool barrier() {
    cg::this_cluster().sync();
    ++barriers;
    return true;
  }
  __device__ void publish(int par, float v, int idx) {  // threads 0 .. P-1 of one warp
    const int t = threadIdx.x;
    if (t < P) *cg::this_cluster().map_shared_rank(mail + par * 16 + me, t) = make_float2(v, __int_as_float(idx));
  }
  __device__ float2 candidate(int par, int r) const { return mail[par * 16 + r]; }
  __device__ const uint4* remote(unsigned off, int rank) const {
    return reinterpret_cast<const uint4*>(cg::this_cluster().map_shared_rank(svd_smem + off, rank));
  }
};

// Barrier of a co-resident (cooperative) grid.  A wait that does not end
// within about two seconds sets the abort flag, which ends every other wait: a
// CTA whose wait was given up leaves the kernel, which reports MPS_ETIMEOUT.
// (A CTA that still finds all others arrived goes on to its next barrier.)
struct GridSync {
  unsigned count, gen, abort, pad;
};

struct GridTeam {
  static constexpr bool kGlobalA = true;
  int me, P;
  GridSync* sync;
  float2* mail;  // global memory: [2][P]
  __device__ bool barrier() {
    __threadfence();
    __syncthreads();
    __shared__ int s_gave_up;
    if (threadIdx.x == 0) {
      int gave_up = 0;
      volatile unsigned* gen = &sync->gen;
      const unsigned g = *gen;
      if (atomicAdd(&sync->count, 1u) == (unsigned)P - 1) {
        sync->count = 0;
        __threadfence();
        atomicAdd(&sync->gen, 1u);
      } else {
        const long long t0 = clock64();
        while (*gen == g) {
          if (clock64() - t0 > 4000000000ll || *(volatile unsigned*)&sync->abort) {
            atomicExch(&sync->abort, 1u);
            gave_up = 1;
            break;
          }
          __nanosleep(20);
        }
      }
      s_gave_up = gave_up;
      __threadfence();
    }
    __syncthreads();
    return !s_gave_up;
  }
  __device__ void publish(int par, float v, int idx) {
    if (threadIdx.x == 0) __stcg(mail + par * P + me, make_float2(v, __int_as_float(idx)));
  }
  __device__ float2 candidate(int par, int r) const { return __ldcg(mail + par * P + r); }
};

// ---- the product C V^H -------------------------------------------------------
// W = C V^H for the kept rows V = B~_{q+1} (k x n): B~_q = W / ||s[:k]|| (Eq.
// Bl, G3), and s_j = ||lam W[:, j]||: the norms of the swept columns carry the
// sweeps' accumulated rounding (a double-float rotation is unitary to about
// 2^-47, some 3e-13 after ten sweeps of 124 columns; FP64 ones leave 2e-14
// after ten of 232), while here the error of a row enters squared: 3e-15.
// 16-column tiles of W are dealt to the CTAs; a tile row runs 2 (or, for few
// threads, 4) outputs per thread over K steps of 16.
constexpr int kPK = 16, kPN = 16, kPM = 64;
constexpr size_t kProductTileBytes = (size_t)(kPM + kPK) * 20 * 16 + 16 * 16 * sizeof(double);
// Dynamic shared memory a CTA can have (the device's 227 KB less the kernels'
// static part); the number of CTAs a theta gets depends on its sizes and this
// alone, so a gate's arithmetic does not depend on the launch it runs in.
constexpr size_t kSvdSmemLimit = 232448 - 1024;

// ---- layout -----------------------------------------------------------------
__host__ __device__ constexpr size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

// Dynamic shared memory of one CTA: the columns, then the per-column arrays.
template <class A>
struct SvdSmem {
  size_t nrm, sg, srt, rnk, na, fl, cls, total;
  // bytes of the column area when P CTAs share an m x n theta; a_smem: A's
  // columns in shared memory (with a copy of the pivot column when P > 1),
  // x_smem: X's blocks too
  __host__ __device__ static size_t col_bytes(int m, int n, int P, bool a_smem, bool x_smem) {
    const size_t ca = (size_t)A::ld(m) * A::kBytes, cx = (size_t)A::ld(n) * A::kBytes;
    const size_t nloc = ((size_t)n + P - 1) / P;
    const size_t r = m < n ? m : n;
    const size_t b = (r + 2 * P - 1) / (2 * P);
    size_t x = x_smem ? (P == 1 ? r : 2 * b) * cx : 0;
    size_t a = a_smem ? (nloc + (P > 1 ? 1 : 0)) * ca : 0;
    if (P == 1) {
      a += x;  // one CTA writes X beside A, and keeps a copy of C where it fits
      if (SvdSmem(align16(a + n * ca), n).total <= kSvdSmemLimit) a += n * ca;
    } else {
      a = a > x ? a : x;
    }
    return align16(a > kProductTileBytes ? a : kProductTileBytes);
  }
  // one CTA: the copy of C fits
  __host__ __device__ static bool has_copy(int m, int n) {
    const size_t ca = (size_t)A::ld(m) * A::kBytes, cx = (size_t)A::ld(n) * A::kBytes;
    return SvdSmem(align16(2 * n * ca + (m < n ? m : n) * cx), n).total <= kSvdSmemLimit;
  }
  // allocation for one CTA and every theta within the capacities
  __host__ __device__ static size_t bytes_one(int mcap, int ncap) {
    return has_copy(mcap, ncap) ? bytes(mcap, ncap, 1, true, true) : kSvdSmemLimit;
  }
  __host__ __device__ SvdSmem(size_t col, int n) {
    nrm = align16(col);
    sg = align16(nrm + 2 * sizeof(float) * n);
    srt = align16(sg + sizeof(double) * n);
    rnk = align16(srt + sizeof(float) * n);
    na = align16(rnk + sizeof(int) * n);
    fl = align16(na + sizeof(double) * n);
    cls = align16(fl + n);
    total = align16(cls + n);
  }
  __host__ __device__ static size_t bytes(int m, int n, int P, bool a_smem, bool x_smem) {
    return SvdSmem(col_bytes(m, n, P, a_smem, x_smem), n).total;
  }
};

// Global workspace of one theta: X's home columns, their norms and flags, the
// grid team's exchange and (global A) A's columns.
template <class A>
struct SvdWs {
  size_t x, nrm, na, fl, stat, mail, a, total;
  __host__ __device__ SvdWs(int m, int n, bool a_global) {
    x = 0;
    nrm = align16((size_t)A::ld(n) * A::kBytes * (size_t)(m < n ? m : n));
    na = align16(nrm + sizeof(double) * n);
    fl = align16(na + sizeof(double) * n);
    stat = align16(fl + n);
    mail = align16(stat + 2 * 256 * sizeof(float2));
    a = align16(mail + 2 * 256 * sizeof(float2));
    total = a + (a_global ? align16((size_t)A::ld(m) * A::kBytes * n) : 0);
  }
};

// Entries of a column that a lane holds in registers at a time: four give the
// rotation eight independent chains.
constexpr int kHold = 4;

// Columns up to which the sweeps take full Gram terms from the start.
constexpr int kHeadsCols = 24;

// log2 of the lanes per column, 3 to 5.  A step's critical path is its column
// length over the lanes, and one warp alone reaches about 60 % of a
// scheduler's FP32 rate: as many lanes as keep 12 warps at work, but no more
// than the column has entries (angle and reductions cost every group the
// same, so further warps only repeat them; 34 columns: 8, 12, 16 warps 852,
// 730, 735 us).  FP64 work fills the SM's two FP64 units from any warp: the
// fewest lanes.  The same for every block size, and so are the sums.
template <class A> __device__ __forceinline__ int lanes_log2(int items, int len) {
  constexpr int cap = 32 * (std::is_same<A, ArF64>::value ? 1 : 12);
  int lg = 5;
  while (lg > 3 && ((items << lg) > cap || (1 << (lg - 1)) >= len)) --lg;
  return lg;
}

// Largest value and its lowest index over nrm[0 .. n) (non-negative floats
// order as integers; dead columns hold -1), the same in every lane.
__device__ __forceinline__ void warp_argmax(const float* nrm, int n, float& best, int& idx) {
  const int lane = threadIdx.x & 31;
  int v = -1, at = 0x7fffffff;
  for (int c = lane; c < n; c += 32) {
    const int x = __float_as_int(nrm[c]);
    if (x > v) {
      v = x;
      at = c;
    }
  }
  const int mx = __reduce_max_sync(0xffffffffu, v);
  idx = __reduce_min_sync(0xffffffffu, v == mx ? at : 0x7fffffff);
  best = mx < 0 ? -1.f : __int_as_float(mx);
}

template <class S, class F> __device__ __forceinline__ S group_sum(S x, int G, F add) {
  for (int o = G >> 1; o > 0; o >>= 1) x = add(x, o);
  return x;
}

template <class A, bool kG>
__device__ __forceinline__ void load_hold(typename A::V (&v)[kHold], typename Mem<kG>::H col, int ld, int len, int r0,
                                          int G) {
#pragma unroll
  for (int i = 0; i < kHold; ++i) {
    const int r = r0 + i * G;
    v[i] = r < len ? A::template load<kG>(col, ld, r) : A::zero_entry();
  }
}
// Entries of a held column in use, the same for every lane.
__device__ __forceinline__ int held_count(int len, int G) { return min(kHold, (len + G - 1) / G); }
template <class A, bool kG>
__device__ __forceinline__ void store_hold(const typename A::V (&v)[kHold], typename Mem<kG>::H col, int ld, int len,
                                           int r0, int G) {
#pragma unroll
  for (int i = 0; i < kHold; ++i) {
    const int r = r0 + i * G;
    if (r < len) A::template store<kG>(col, ld, r, v[i]);
  }
}

// ---- one pair ---------------------------------------------------------------
struct PairStat {
  float off2 = 0.f;  // largest |g|^2 / (a b) met
  int sig = 0;       // a rotation above the stopping tolerance
};

// One step on the columns x, y (length len) by the G lanes of a group; every
// lane of the warp calls it (act false: the group has no pair and only keeps
// the shuffles in step).  Returns whether the pair was rotated.
template <class A, bool kG, bool kHeads>
__device__ __forceinline__ bool jacobi_pair(typename Mem<kG>::H cx, typename Mem<kG>::H cy, int ld, int len, int gl,
                                            int G, bool act, typename A::S& na, typename A::S& nb, float rot2,
                                            float sig2, PairStat& st, bool& significant) {
  using S = typename A::S;
  using V = typename A::V;
  V x[kHold], y[kHold];
  load_hold<A, kG>(x, cx, ld, len, gl, G);
  load_hold<A, kG>(y, cy, ld, len, gl, G);
  const int step = kHold * G, nh = held_count(len, G);
  S gr, gi;
  if constexpr (kHeads) {
    float re = 0.f, im = 0.f;
    auto head_dot = [&](const V(&u)[kHold], const V(&v)[kHold]) {
#pragma unroll
      for (int i = 0; i < kHold; ++i) {
        const float2 a = A::head(u[i]), b = A::head(v[i]);
        re = fmaf(a.x, b.x, fmaf(a.y, b.y, re));
        im = fmaf(a.x, b.y, fmaf(-a.y, b.x, im));
      }
    };
    head_dot(x, y);
    for (int r0 = gl + step; r0 - gl < len; r0 += step) {
      V u[kHold], v[kHold];
      load_hold<A, kG>(u, cx, ld, len, r0, G);
      load_hold<A, kG>(v, cy, ld, len, r0, G);
      head_dot(u, v);
    }
    for (int o = G >> 1; o > 0; o >>= 1) {
      re += __shfl_xor_sync(0xffffffffu, re, o);
      im += __shfl_xor_sync(0xffffffffu, im, o);
    }
    gr = A::zero();
    gi = gr;
    if constexpr (A::kRough) {
      gr.h = re;
      gi.h = im;
    }
  } else {
    typename A::Acc acc;
#pragma unroll
    for (int i = 0; i < kHold; ++i)
      if (i < nh) A::dot(acc, x[i], y[i]);
    for (int r0 = gl + step; r0 - gl < len; r0 += step) {
      V u[kHold], v[kHold];
      load_hold<A, kG>(u, cx, ld, len, r0, G);
      load_hold<A, kG>(v, cy, ld, len, r0, G);
#pragma unroll
      for (int i = 0; i < kHold; ++i) A::dot(acc, u[i], v[i]);
    }
    A::dot_sum(acc, G, gr, gi);
  }
  const float off2 = act ? A::off2(na, nb, gr, gi) : 0.f;
  st.off2 = fmaxf(st.off2, off2);
  bool rot = off2 > rot2;
  significant = off2 > sig2;
  if (!__any_sync(0xffffffffu, rot)) return false;
  if constexpr (!kHeads) {
    // nearly equal norms: the angle needs their difference, so both afresh
    const float fa = A::to_float(na), fb = A::to_float(nb);
    const bool close = rot && fabsf(fa - fb) <= 0.00390625f * fmaxf(fa, fb);
    if (__any_sync(0xffffffffu, close)) {
      typename A::NAcc xa, ya;
      for (int r = gl; r < len; r += G) {
        A::nrm(xa, A::template load<kG>(cx, ld, r));
        A::nrm(ya, A::template load<kG>(cy, ld, r));
      }
      S sa, sb;
      A::norm2_sum(xa, ya, G, sa, sb);
      if (close) {
        na = sa;
        nb = sb;
      }
    }
  }
  Rot<S> o;
  if (rot) rot = A::angle(na, nb, gr, gi, o);
  if (rot) {
    const auto k = A::rot_const(o);
#pragma unroll
    for (int i = 0; i < kHold; ++i)
      if (i < nh) A::rotate(k, x[i], y[i]);
    store_hold<A, kG>(x, cx, ld, len, gl, G);
    store_hold<A, kG>(y, cy, ld, len, gl, G);
    for (int r0 = gl + step; r0 < len; r0 += step) {
      load_hold<A, kG>(x, cx, ld, len, r0, G);
      load_hold<A, kG>(y, cy, ld, len, r0, G);
#pragma unroll
      for (int i = 0; i < kHold; ++i) A::rotate(k, x[i], y[i]);
      store_hold<A, kG>(x, cx, ld, len, r0, G);
      store_hold<A, kG>(y, cy, ld, len, r0, G);
    }
    na = A::sub(na, o.dn);
    nb = A::add(nb, o.dn);
    st.sig |= significant ? 1 : 0;
  }
  return rot;
}

// ---- the SVD ------------------------------------------------------------------
// Every thread of every CTA of the team calls it.  gws: the global workspace
// (SvdWs).  C and lam_l are read past L1: a run of gates changes them between
// calls.  The dynamic shared memory holds an SvdSmem of the team's size.  kGX: X's blocks stay in the
// global workspace.  Writes B~_{q+1} (k x n), lam_{q+1}, *chi_out and the
// report; returns k, or 0 when a barrier was given up.  Bq (nullable): B~_q = C V^H / ||s[:k]|| as well.
template <class A, class R, class Team, bool kGX>
__device__ int svd_body(Team& tm, const cplx<R>* __restrict__ Cm, const double* __restrict__ lam_l, int m, int n,
                        const SvdParams& p, cplx<R>* __restrict__ Bnext, double* __restrict__ lam_next, int* chi_out,
                        DevReport* __restrict__ rep, cplx<R>* __restrict__ Bq, char* __restrict__ gws) {
  using S = typename A::S;
  using V = typename A::V;
  constexpr bool kGA = Team::kGlobalA;
  const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31;
  const int me = tm.me, P = tm.P;
  const int lda = A::ld(m), ldx = A::ld(n);
  const size_t ca = (size_t)lda * A::kBytes, cx = (size_t)ldx * A::kBytes;
  const int rmax = min(m, n);
  const SvdWs<A> W(m, n, kGA);
  const SvdSmem<A> L(SvdSmem<A>::col_bytes(m, n, P, !kGA, !kGX), n);
  char* gx = gws + W.x;
  // one CTA: X follows A's n columns in shared memory
  const unsigned x0 = std::is_same<Team, OneTeam>::value ? (unsigned)(n * ca) : 0u;
  // and conj(C) 2^-ec follows X where it fits
  const bool direct = std::is_same<Team, OneTeam>::value && SvdSmem<A>::has_copy(m, n);
  const unsigned c0 = x0 + (unsigned)(rmax * cx);
  double* gnrm = reinterpret_cast<double*>(gws + W.nrm);
  double* gna = reinterpret_cast<double*>(gws + W.na);
  unsigned char* gfl = reinterpret_cast<unsigned char*>(gws + W.fl);
  float2* gstat = reinterpret_cast<float2*>(gws + W.stat);
  using HA = typename Mem<kGA>::H;
  using HX = typename Mem<kGX>::H;
  auto acol = [&](int i, int c) -> HA {  // column c of A, at local place i
    if constexpr (kGA)
      return gws + W.a + (size_t)c * ca;
    else
      return (unsigned)(i * ca);
  };
  float* nrm = reinterpret_cast<float*>(svd_smem + L.nrm);
  double* sg = reinterpret_cast<double*>(svd_smem + L.sg);
  float* srt = reinterpret_cast<float*>(svd_smem + L.srt);
  int* rnk = reinterpret_cast<int*>(svd_smem + L.rnk);
  S* nA = reinterpret_cast<S*>(svd_smem + L.na);
  unsigned char* fl = svd_smem + L.fl;
  unsigned char* cls = svd_smem + L.cls;
  __shared__ int s_i[4];
  __shared__ float s_f[4];
  __shared__ double s_d[4];
  auto addS = [](S x, int o) { return A::shfl_add(x, o); };
  const long long t_start = clock64();

  // ---- scale (exponents only; the same for every CTA)
  const int nloc = (n - me + P - 1) / P;  // columns me, me + P, ... of A
  if (tid == 0) s_i[0] = s_i[1] = -100000;
  __syncthreads();
  // small thetas are read once and held in registers
  constexpr int kKeep = 2;
  const bool keep = m * nloc <= kKeep * T;
  cplx<R> zk[kKeep];
  double lk[kKeep];
  {
    int emax = -100000, cmax = -100000;
    auto look = [&](const cplx<R> z, double lam) {
      const int el = ((__double2hiint(lam) >> 20) & 0x7ff) - 1023;
      int ez;
      if constexpr (sizeof(R) == 8) {
        ez = max((__double2hiint(z.x) >> 20) & 0x7ff, (__double2hiint(z.y) >> 20) & 0x7ff) - 1023;
      } else {
        ez = max((__float_as_int(z.x) >> 23) & 0xff, (__float_as_int(z.y) >> 23) & 0xff) - 127;
      }
      emax = max(emax, el + ez);
      cmax = max(cmax, ez);
    };
    if (keep) {
#pragma unroll
      for (int i = 0; i < kKeep; ++i) {
        const int t = tid + i * T;
        if (t < m * nloc) {
          const int r = t / nloc;
          zk[i] = __ldcg(Cm + (size_t)r * n + me + (t - r * nloc) * P);
          lk[i] = __ldcg(lam_l + (r >> 1));
          look(zk[i], lk[i]);
        }
      }
    } else {
      for (int t = tid; t < m * nloc; t += T) {
        const int r = t / nloc;
        look(__ldcg(Cm + (size_t)r * n + me + (t - r * nloc) * P), __ldcg(lam_l + (r >> 1)));
      }
    }
    emax = __reduce_max_sync(0xffffffffu, emax);
    cmax = __reduce_max_sync(0xffffffffu, cmax);
    if (lane == 0) {
      atomicMax(&s_i[0], emax);
      atomicMax(&s_i[1], cmax);
    }
  }
  __syncthreads();
  if constexpr (!std::is_same<Team, OneTeam>::value) {
    if (tid < 32) tm.publish(0, (float)s_i[1], s_i[0]);
    if (!tm.barrier()) return 0;
    int e = -100000;
    float c = -100000.f;
    for (int r = 0; r < P; ++r) {
      const float2 v = tm.candidate(0, r);
      e = max(e, __float_as_int(v.y));
      c = fmaxf(c, v.x);
    }
    __syncthreads();
    if (tid == 0) {
      s_i[0] = e;
      s_i[1] = (int)c;
    }
    __syncthreads();
  }
  const int ex = max(-900, min(900, s_i[0] - kScaleExp));
  const int ec = max(-900, min(900, s_i[1]));                             // exponent of the largest entry of C
  const double scl = __longlong_as_double((long long)(1023 - ex) << 52);   // 2^-ex
  const double cscl = __longlong_as_double((long long)(1023 - ec) << 52);  // 2^-ec

  // ---- load this CTA's columns of A and their squared norms
  auto place = [&](int t, const cplx<R> z, double lam) {
    const int r = t / nloc, i = t - r * nloc;
    const double w = lam * scl;
    A::template store<kGA>(acol(i, me + i * P), lda, r, A::make(w * double(z.x), w * double(z.y)));
    if (direct)
      A::template store<false>(c0 + (unsigned)(i * ca), lda, r, A::make(cscl * double(z.x), -cscl * double(z.y)));
  };
  if (keep) {
#pragma unroll
    for (int i = 0; i < kKeep; ++i)
      if (tid + i * T < m * nloc) place(tid + i * T, zk[i], lk[i]);
  } else {
    for (int t = tid; t < m * nloc; t += T) {
      const int r = t / nloc;
      place(t, __ldcg(Cm + (size_t)r * n + me + (t - r * nloc) * P), __ldcg(lam_l + (r >> 1)));
    }
  }
  __syncthreads();
  {
    const int lg = lanes_log2<A>(nloc, m), G = 1 << lg, gl = tid & (G - 1), grp = tid >> lg, NG = T >> lg;
    for (int i0 = 0; i0 < nloc; i0 += NG) {
      const int i = i0 + grp;
      const int ii = i < nloc ? i : 0;
      const HA col = acol(ii, me + ii * P);
      float v = 0.f;
      for (int r = gl; r < m; r += G) v += A::head_norm2(A::template load<kGA>(col, lda, r));
      for (int o = G >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (gl == 0 && i < nloc) nrm[i] = v;
    }
  }
  __syncthreads();
  const long long t_load = clock64();

  // ---- pivoted modified Gram-Schmidt.  Column j of X gets X[c, j] =
  // conj(q_j^H a_c): the rows of R in the original column order, so no
  // permutation is undone later.  The residual norms pick the pivot and stop
  // the factorisation at the noise floor (4 u ||A||_F, or less when the
  // truncation threshold is lower): what is left changes squared singular
  // values by its own square only.
  const float cut_rel = (float)fmin(4.0 * A::unit(), 0.125 * p.trunc_rel);
  float fro2 = 0.f;
  int r = 0;
  {
    const int lg = lanes_log2<A>(nloc, m), G = 1 << lg, gl = tid & (G - 1), grp = tid >> lg, NG = T >> lg;
    if constexpr (!std::is_same<Team, OneTeam>::value) {
      // Frobenius norm over the team
      if (tid < 32) {
        float f = 0.f;
        for (int i = lane; i < nloc; i += 32) f += nrm[i];
        f = warp_sum(f);
        tm.publish(1, f, 0);
      }
      if (!tm.barrier()) return 0;
      for (int k = 0; k < P; ++k) fro2 += tm.candidate(1, k).x;
    } else {
      float f = 0.f;
      for (int i = lane; i < nloc; i += 32) f += nrm[i];
      fro2 = warp_sum(f);
    }
    const float stop2 = fmaxf(kZeroNorm2, cut_rel * cut_rel * fro2);
    // Without a truncation threshold every nonzero direction is kept (the rows
    // of B~_{q+1} then span those of the unscaled C, which keeps B~_q
    // right-canonical on the rows that lam_q weighs with rounding noise): residuals
    // that count as zero columns are scaled up to just above them, at most 4e-17
    // of the largest entry, a perturbation of A below its rounding, and the
    // factorisation goes on.
    const bool keep_noise = p.trunc_rel == 0.0;
    for (int j = 0; j < rmax;) {
      float* nc = nrm + (j & 1) * n;
      float* nn = nrm + ((j & 1) ^ 1) * n;
      float best;
      int li;  // local index of the pivot at its owner
      int owner = 0;
      if constexpr (std::is_same<Team, OneTeam>::value) {
        warp_argmax(nc, nloc, best, li);
      } else {
        if (tid < 32) {
          warp_argmax(nc, nloc, best, li);
          tm.publish(j & 1, best, li);
        }
        if (!tm.barrier()) return 0;
        best = -1.f;
        li = 0;
        for (int k0 = 0; k0 < P; k0 += 32) {
          const float2 cd = k0 + lane < P ? tm.candidate(j & 1, k0 + lane) : make_float2(-1.f, 0.f);
          const int mx = __reduce_max_sync(0xffffffffu, __float_as_int(cd.x));
          const unsigned who = __ballot_sync(0xffffffffu, __float_as_int(cd.x) == mx);
          const int w = __ffs(who) - 1;
          if (mx >= 0 && __int_as_float(mx) > best) {
            best = __int_as_float(mx);
            owner = k0 + w;
            li = __float_as_int(__shfl_sync(0xffffffffu, cd.y, w));
          }
        }
      }
      if (!(best > stop2)) {
        if (!keep_noise || !(best > 0.f)) break;
        const float up = pow2f(max(1, min(60, (exp_of(stop2) - exp_of(best)) / 2 + 1)));
        for (int t = tid; t < m * nloc; t += T) {
          const int i = t / m, rr = t - i * m;
          if (nc[i] < 0.f) continue;
          const HA col = acol(i, me + i * P);
          A::template store<kGA>(col, lda, rr, A::times(A::template load<kGA>(col, lda, rr), up));
        }
        __syncthreads();
        for (int i = tid; i < nloc; i += T)
          if (nc[i] >= 0.f) nc[i] *= up * up;
        if (!tm.barrier()) return 0;
        continue;
      }
      const int pc = owner + li * P;  // pivot column of A
      HA pcol = acol(li, pc);
      if constexpr (std::is_same<Team, ClusterTeam>::value) {
        if (owner != me) {
          const unsigned copy = (unsigned)(((n + P - 1) / P) * ca);
          const uint4* src = tm.remote(pcol, owner);
          for (int t = tid; t < (int)(ca / 16); t += T) reinterpret_cast<uint4*>(svd_smem + copy)[t] = src[t];
          pcol = copy;
        }
        __syncthreads();
      }
      // the pivot's norm, then per column: dot product with the pivot, its
      // share subtracted, the new residual norm
      V px[kHold];
      const int step = kHold * G, nh = held_count(m, G);
      S p2 = A::zero(), pinv = p2, pinv2 = p2;  // |p|^2, 1 / |p|, 1 / |p|^2
      bool have_p = false;
      auto put = [&](int c, V v) {  // X[c, j]
        if constexpr (std::is_same<Team, OneTeam>::value)
          A::template store<false>((unsigned)(x0 + j * cx), ldx, c, v);
        else
          A::template store<true>(gx + (size_t)j * cx, ldx, c, v);
      };
      for (int i0 = 0; i0 < nloc; i0 += NG) {
        const int i = i0 + grp;
        const int c = me + i * P;
        const bool in = i < nloc;
        const bool alive = in && nc[in ? i : 0] >= 0.f && c != pc;
        if (__any_sync(0xffffffffu, alive || (in && c == pc))) {
          const HA col = alive ? acol(i, c) : pcol;
          V y[kHold];
          typename A::NAcc pn;
          if (!have_p) {
            load_hold<A, kGA>(px, pcol, lda, m, gl, G);
#pragma unroll
            for (int t = 0; t < kHold; ++t)
              if (t < nh) A::nrm(pn, px[t]);
            for (int rr = gl + step; rr < m; rr += G) A::nrm(pn, A::template load<kGA>(pcol, lda, rr));
          }
          load_hold<A, kGA>(y, col, lda, m, gl, G);
          typename A::Acc acc;
#pragma unroll
          for (int t = 0; t < kHold; ++t)
            if (t < nh) A::dot(acc, px[t], y[t]);
          for (int rr = gl + step; rr < m; rr += G)
            A::dot(acc, A::template load<kGA>(pcol, lda, rr), A::template load<kGA>(col, lda, rr));
          S dr, di;
          if (!have_p) {
            have_p = true;
            A::dot_norm_sum(acc, pn, G, dr, di, p2);
            pinv = A::rsqrt(p2);
            pinv2 = A::mul(pinv, pinv);
          } else {
            A::dot_sum(acc, G, dr, di);
          }
          float v = 0.f;
          if (alive) {
            const auto k = A::axpy_const(A::mul(dr, pinv2), A::mul(di, pinv2));
#pragma unroll
            for (int t = 0; t < kHold; ++t)
              if (t < nh) {
                y[t] = A::axpy(k, px[t], y[t]);
                v += A::head_norm2(y[t]);
              }
            store_hold<A, kGA>(y, col, lda, m, gl, G);
            for (int rr = gl + step; rr < m; rr += G) {
              const V z = A::axpy(k, A::template load<kGA>(pcol, lda, rr), A::template load<kGA>(col, lda, rr));
              A::template store<kGA>(col, lda, rr, z);
              v += A::head_norm2(z);
            }
          }
          for (int o = G >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (alive && gl == 0) {
            nn[i] = v;
            put(c, A::cval(A::mul(dr, pinv), A::sub(A::zero(), A::mul(di, pinv))));
          }
        }
        if (in && !alive && gl == 0) {
          nn[i] = -1.f;
          put(c, A::cval(c == pc ? A::mul(p2, pinv) : A::zero(), A::zero()));
        }
      }
      r = ++j;
      __syncthreads();
    }
  }
  if (r == 0) {
    // a zero theta: one unit row with a zero singular value (NaN for a theta
    // that holds infinities or NaN)
    if (me == 0) {
      const double z = fro2 - fro2;
      for (int c = tid; c < n; c += T) Bnext[c] = cmk<R>(R(c == 0 ? 1.0 + z : z), R(0));
      if (Bq)
        for (int row = tid; row < m; row += T) Bq[row] = __ldcg(Cm + (size_t)row * n);
      if (tid == 0) {
        lam_next[0] = z;
        *chi_out = 1;
        if (0.0 < rep->min_kept_sv) rep->min_kept_sv = 0.0;
        rep->two_qubit_gates += 1;
        rep->inv_norm = 1.0;
      }
    }
    return 1;
  }
  const long long t_gs = clock64();

  // ---- blocks of X
  const int b = P == 1 ? r : (r + 2 * P - 1) / (2 * P);  // P == 1: one block of all columns
  const int M = 2 * P - 1;
  const int nslots = P == 1 ? 1 : 2;
  auto block_at = [&](int slot, int rnd) -> int {
    const int pos = slot == 0 ? me : M - me;
    if (pos == 0) return 0;
    return 1 + ((pos - 1 - rnd) % M + M) % M;
  };
  // the column held at local place i, with column id `id`
  auto held = [&](int i, int id) -> HX {
    if constexpr (kGX)
      return gx + (size_t)id * cx;
    else
      return (unsigned)(x0 + i * cx);
  };
  auto fetch = [&](int slot, int blk) {  // home -> slot
    if constexpr (!kGX) {
      const int cnt = max(0, min(b, r - blk * b));
      const size_t u = (size_t)cnt * cx / 16;
      const uint4* src = reinterpret_cast<const uint4*>(gx + (size_t)blk * b * cx);
      uint4* dst = reinterpret_cast<uint4*>(svd_smem + (size_t)slot * b * cx);
      for (size_t t = tid; t < u; t += T) dst[t] = __ldcg(src + t);
    }
  };
  auto flush = [&](int slot, int blk) {  // slot -> home, with the norms and flags
    const int cnt = max(0, min(b, r - blk * b));
    if constexpr (!kGX) {
      const size_t u = (size_t)cnt * cx / 16;
      const uint4* src = reinterpret_cast<const uint4*>(svd_smem + (size_t)slot * b * cx);
      uint4* dst = reinterpret_cast<uint4*>(gx + (size_t)blk * b * cx);
      for (size_t t = tid; t < u; t += T) __stcg(dst + t, src[t]);
    }
    for (int t = tid; t < cnt; t += T) {
      const int id = blk * b + t;
      S v = nA[id];
      double d = 0.0;
      memcpy(&d, &v, sizeof(S));
      __stcg(gna + id, d);
      __stcg(gfl + id, fl[id]);
    }
  };
  auto fetch_meta = [&](int blk) {
    const int cnt = max(0, min(b, r - blk * b));
    for (int t = tid; t < cnt; t += T) {
      const int id = blk * b + t;
      const double d = __ldcg(gna + id);
      S v;
      memcpy(&v, &d, sizeof(S));
      nA[id] = v;
      fl[id] = __ldcg(gfl + id);
    }
  };
  if (!tm.barrier()) return 0;  // X complete (and, with several CTAs, A's shared memory free)
  if (P > 1)
    for (int slot = 0; slot < nslots; ++slot) fetch(slot, block_at(slot, 0));
  for (int id = tid; id < r; id += T) fl[id] = 2;  // bit 0: rotated in this sweep, bit 1: in the previous one
  __syncthreads();

  // ---- sweeps.  Stopping rule: rotate while |g| > tol sqrt(a b), tol = 4
  // sqrt(max(m, n)) u; a sweep without such a rotation ends them.  Pairs down
  // to u are still rotated when they are met (the kept rows' orthogonality),
  // without asking for another sweep.
  const float tol_sig = p.tol > 0 ? (float)p.tol : (float)(4.0 * sqrt((double)max(m, n)) * A::unit());
  const float tol_rot = p.tol > 0 ? (float)p.tol : (float)A::unit();
  const float tol_heads = fmaxf(4e-6f, tol_sig);
  // the pair step compares squares
  const float sig2 = tol_sig * tol_sig, rot2 = tol_rot * tol_rot, heads2 = tol_heads * tol_heads;
  const int kcap = min(p.chi_max, rmax);
  const double trunc2 = p.trunc_rel * p.trunc_rel;
  const float thr_rel2 = (float)trunc2;
  int sweep = 0;
  // (few columns: the full Gram terms cost little more than the heads, and a
  // sweep less is run)
  bool converged = false, heads = A::kRough && r > kHeadsCols, prev_full = false;
  for (;; ++sweep) {
    // squared norms of this CTA's columns, to everyone
    {
      const int items = nslots * b;
      const int lg = lanes_log2<A>(items, n), G = 1 << lg, gl = tid & (G - 1), grp = tid >> lg, NG = T >> lg;
      for (int i0 = 0; i0 < items; i0 += NG) {
        const int i = i0 + grp, slot = i >= b ? 1 : 0, c = i - slot * b;
        const int blk = block_at(slot, 0), id = blk * b + c;
        const bool ok = i < items && id < r;
        if (!__any_sync(0xffffffffu, ok)) continue;
        const HX col = held(ok ? i : 0, ok ? id : 0);
        typename A::NAcc acc;
        if (ok)
          for (int rr = gl; rr < n; rr += G) A::nrm(acc, A::template load<kGX>(col, ldx, rr));
        const S v = group_sum(A::nrm_value(acc), G, addS);
        if (ok && gl == 0) {
          nA[id] = v;
          const double d = A::to_double(v);
          if (P == 1) {
            sg[id] = d;
            nrm[id] = A::to_float(v);
          } else
            __stcg(gnrm + id, d);
        }
      }
    }
    if (!tm.barrier()) return 0;
    if (P > 1)
      for (int id = tid; id < r; id += T) sg[id] = __ldcg(gnrm + id);
    if (sweep > 0) {
      // the previous sweep's verdict: largest coupling met, and whether a
      // rotation above the tolerance was made
      float off = 0.f, sig = 0.f;  // off: squared
      if (P == 1) {
        off = s_f[0];
        sig = s_f[1];
      } else {
        for (int k = 0; k < P; ++k) {
          const float2 v = __ldcg(gstat + (sweep & 1) * 256 + k);
          off = fmaxf(off, v.x);
          sig = fmaxf(sig, v.y);
        }
      }
      if (!heads && sig == 0.f) converged = true;
      // heads (errors of about 1e-7) resolve couplings above 4e-6: once a
      // sweep met none above 1e-3 the next one finds about their squares
      prev_full = !heads;
      if (heads && off < 1e-6f) heads = false;
    }
    __syncthreads();
    if (converged || sweep >= p.max_sweeps) break;
    // ---- tail: T = the smallest columns, all outside the kept set, whose
    // total weight is at most a quarter of the next larger column's and, when
    // the threshold and not chi_max decides the cut, of the threshold's.
    // Every singular value of the T block is then at most half of every other
    // column's norm and of the threshold, so once the other columns are
    // orthogonal to each other and to T they hold the leading singular vectors
    // whatever T looks like: pairs inside T are left alone (the discarded
    // weight is the sum).
    if (P > 1) {
      for (int id = tid; id < r; id += T) nrm[id] = (float)sg[id];
      __syncthreads();
    }
    if (tid == 0) {
      s_i[0] = 0;
      s_i[1] = r;
      s_f[0] = 0.f;
      s_f[1] = 0.f;
    }
    // every warp for itself: the largest norm, the columns above the threshold
    // and the weight of the rest.  When the threshold decides the cut that
    // weight alone settles T (all of the rest, or nothing for few columns)
    int vm = 0, above = 0;
    float rest = 0.f;
    for (int id = lane; id < r; id += 32) vm = max(vm, __float_as_int(nrm[id]));
    const float thr = thr_rel2 * __int_as_float(__reduce_max_sync(0xffffffffu, vm));
    for (int id = lane; id < r; id += 32) {
      const float v = nrm[id];
      above += v > thr;
      rest += v > thr ? 0.f : v;
    }
    above = __reduce_add_sync(0xffffffffu, above);
    rest = warp_sum(rest);
    const bool all_rest = above <= kcap && rest <= 0.25f * thr;
    if (all_rest || r <= 32) {
      __syncthreads();
      for (int id = tid; id < r; id += T) {
        const unsigned char c = all_rest && !(nrm[id] > thr) ? 1 : 0;
        if (sweep > 0 && c != cls[id]) fl[id] |= 2;  // tested again when it joins or leaves T
        cls[id] = c;
      }
    } else {
    __syncthreads();
    {
      const int lg = lanes_log2<A>(r, r), G = 1 << lg, gl = tid & (G - 1), grp = tid >> lg, NG = T >> lg;
      for (int i0 = 0; i0 < r; i0 += NG) {
        if (!__any_sync(0xffffffffu, i0 + grp < r)) continue;
        const int id = min(i0 + grp, r - 1);
        const float v = nrm[id];
        int rk = 0;
        for (int h = gl; h < r; h += G) {
          const float u = nrm[h];
          rk += (u > v) || (u == v && h < id);
        }
        for (int o = G >> 1; o > 0; o >>= 1) rk += __shfl_xor_sync(0xffffffffu, rk, o);
        rk = min(rk, r - 1);  // NaN norms compare false
        if (gl == 0 && i0 + grp < r) {
          rnk[id] = rk;
          srt[rk] = v;
        }
      }
    }
    __syncthreads();
    {
      const int kept = max(1, min(above, kcap));
      const float lim = above >= kcap ? INFINITY : thr;
      for (int t = tid; t < r; t += T) {
        if (t < kept) continue;
        float w = 0.f;
        for (int h = r - 1; h >= t; --h) w += srt[h];
        if (w <= 0.25f * fminf(lim, srt[t - 1])) atomicMin(&s_i[1], t);
      }
    }
    __syncthreads();
    const int t_first = s_i[1];
    for (int id = tid; id < r; id += T) {
      const unsigned char c = rnk[id] >= t_first ? 1 : 0;
      // a column that joins or leaves T is tested again
      if (sweep > 0 && c != cls[id]) fl[id] |= 2;
      cls[id] = c;
    }
    }
    __syncthreads();

    PairStat st;
    auto step = [&](HX x, HX y, int ix, int iy, bool act, int gl, int G) {
      act = act && !(cls[ix] & cls[iy]);
      // both unchanged since a full sweep tested them: orthogonal still
      if (act && prev_full && !heads && !((fl[ix] | fl[iy]) & 3)) act = false;
      if (!__any_sync(0xffffffffu, act)) return;
      S na = nA[ix], nb = nA[iy];
      bool sig, rot;
      if (A::kRough && heads)
        rot = jacobi_pair<A, kGX, A::kRough>(x, y, ldx, n, gl, G, act, na, nb, heads2, heads2, st, sig);
      else
        rot = jacobi_pair<A, kGX, false>(x, y, ldx, n, gl, G, act, na, nb, rot2, sig2, st, sig);
      if (rot && gl == 0) {
        nA[ix] = na;
        nA[iy] = nb;
        if (sig) {
          fl[ix] |= 1;
          fl[iy] |= 1;
        }
      }
    };
    // Round 0 pairs all columns this CTA holds (circle method over np players),
    // the others pair the columns of its two blocks.
    const int nl = P == 1 ? r : 2 * b;  // columns held
    const int np = nl + (nl & 1), mod = np - 1, pairs = np >> 1;
    const int lg = lanes_log2<A>(pairs, n), G = 1 << lg, gl = tid & (G - 1), grp = tid >> lg, NG = T >> lg;
    for (int rnd = 0; rnd < (P == 1 ? 1 : M); ++rnd) {
      const int b0 = block_at(0, rnd), b1 = block_at(1, rnd);
      const int ns = rnd == 0 ? mod : b;
      for (int sr = 0; sr < ns; ++sr) {
        for (int k0 = 0; k0 < pairs; k0 += NG) {
          const int k = k0 + grp;
          int i0, i1;
          if (rnd == 0) {
            i0 = mod;
            i1 = sr;
            if (k > 0) {
              i0 = sr + k;
              i0 -= i0 >= mod ? mod : 0;
              i1 = sr - k;
              i1 += i1 < 0 ? mod : 0;
            }
          } else {
            i0 = k;
            i1 = k + sr;
            i1 += i1 >= b ? 0 : b;  // b + (k + sr) mod b
          }
          bool act = k < pairs && i0 < nl && i1 < nl;
          if (!act) i0 = i1 = 0;
          int d0 = i0, d1 = i1;  // column ids
          if (P > 1) {
            d0 = i0 < b ? b0 * b + i0 : b1 * b + i0 - b;
            d1 = i1 < b ? b0 * b + i1 : b1 * b + i1 - b;
            act = act && d0 < r && d1 < r;
            if (!act) d0 = d1 = 0;
          }
          step(held(i0, d0), held(i1, d1), d0, d1, act, gl, G);
        }
        __syncthreads();
      }
      if (P == 1) break;
      // hand the blocks on: position pos -> pos + 1 (pos >= 1), 2P - 1 -> 1
      for (int slot = 0; slot < 2; ++slot)
        if (!(slot == 0 && me == 0)) flush(slot, slot ? b1 : b0);
      if (!tm.barrier()) return 0;
      for (int slot = 0; slot < 2; ++slot)
        if (!(slot == 0 && me == 0)) {
          const int nb = block_at(slot, rnd + 1);
          fetch(slot, nb);
          fetch_meta(nb);
        }
      __syncthreads();
    }
    // the sweep's verdict, and the flags roll on
    {
      const int o = __reduce_max_sync(0xffffffffu, __float_as_int(st.off2));
      const int s = __any_sync(0xffffffffu, st.sig);
      if (lane == 0) {
        atomicMax(reinterpret_cast<int*>(&s_f[0]), o);
        if (s) s_f[1] = 1.f;
      }
    }
    __syncthreads();
    if (P == 1 && !heads && s_f[1] == 0.f) {
      // nothing above the tolerance was rotated: the norms stand
      converged = true;
      ++sweep;
      break;
    }
    if (P > 1 && tid == 0) __stcg(gstat + ((sweep + 1) & 1) * 256 + me, make_float2(s_f[0], s_f[1]));
    for (int id = tid; id < r; id += T) fl[id] = (fl[id] & 1) ? 2 : 0;
    __syncthreads();
  }
  const long long t_sw = clock64();

  // ---- squared singular values (in units of 4^ex), ranks (descending, ties by
  // index), truncation
  for (int id = tid; id < r; id += T)
    if (sg[id] <= (double)kZeroNorm2 * 1e-2) sg[id] = 0.0;
  __syncthreads();
  {
    const int lg = lanes_log2<A>(r, r), G = 1 << lg, gl = tid & (G - 1), grp = tid >> lg, NG = T >> lg;
    for (int i0 = 0; i0 < r; i0 += NG) {
      if (!__any_sync(0xffffffffu, i0 + grp < r)) continue;
      const int id = min(i0 + grp, r - 1);
      const long long v = __double_as_longlong(sg[id]);  // non-negative doubles order as integers
      int rk = 0;
      for (int h = gl; h < r; h += G) {
        const long long u = __double_as_longlong(sg[h]);
        rk += (u > v) || (u == v && h < id);
      }
      for (int o = G >> 1; o > 0; o >>= 1) rk += __shfl_xor_sync(0xffffffffu, rk, o);
      if (gl == 0 && i0 + grp < r) rnk[id] = rk;
    }
  }
  __syncthreads();
  // kept count: every warp for itself
  int k;
  {
    long long vmax = 0;
    for (int id = lane; id < r; id += 32) vmax = max(vmax, rnk[id] == 0 ? __double_as_longlong(sg[id]) : 0ll);
    const unsigned who = __ballot_sync(0xffffffffu, vmax != 0);
    vmax = __shfl_sync(0xffffffffu, vmax, who ? __ffs(who) - 1 : 0);
    const long long thr = __double_as_longlong(trunc2 * __longlong_as_double(vmax));
    int cnt = 0;
    for (int id = lane; id < r; id += 32) cnt += __double_as_longlong(sg[id]) > thr;
    k = max(1, min(__reduce_add_sync(0xffffffffu, cnt), kcap));
  }
  // (FP64 sweeps of few columns leave less than the product's own rounding)
  const bool refine = sizeof(R) == 8 && (std::is_same<A, ArDF>::value || n >= 32);
  if (tid >= T - 32 && (me == 0 || !refine)) {
    // 1 / ||s[:k]|| and the report, by the last warp while the others go on;
    // sums and quotients in the sweeps' arithmetic (a chain of FP64 roots and
    // divisions took 5 us of every gate, whatever its size)
    S kept = A::zero(), drop = kept, vmin = kept, vnext = kept;
    for (int id = lane; id < r; id += 32) {
      const S v = A::from_double(sg[id]);
      if (rnk[id] < k)
        kept = A::add(kept, v);
      else
        drop = A::add(drop, v);
      if (rnk[id] == k - 1) vmin = v;
      if (rnk[id] == k) vnext = v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      kept = A::shfl_add(kept, o);
      drop = A::shfl_add(drop, o);
      vmin = A::shfl_add(vmin, o);
      vnext = A::shfl_add(vnext, o);
    }
    // lanes 0, 1, 2: reciprocal roots of the kept weight, s_k^2, the total
    const S total = A::add(kept, drop);
    const S y = lane == 0 ? kept : (lane == 1 ? vmin : total);
    const bool pos = A::to_float(y) > 0.f;
    const S ry = A::rsqrt(pos ? y : A::from_double(1.0));
    const double inv = __shfl_sync(0xffffffffu, A::to_double(ry), 0);
    double out = inv;                                                                  // lane 0
    if (lane == 1) out = pos ? A::to_double(A::mul(y, ry)) * inv : 0.0;                // s_k / ||s[:k]||
    if (lane == 2) out = pos ? A::to_double(A::mul(A::mul(drop, ry), ry)) : 0.0;       // discarded share
    const double ratio = __shfl_sync(0xffffffffu, out, 1), share = __shfl_sync(0xffffffffu, out, 2);
    if (lane == 0) {
      if (!refine) s_d[1] = inv;
      if (me == 0) {
        rep->discarded_weight += share;
        if (!refine && ratio < rep->min_kept_sv) rep->min_kept_sv = ratio;
        if (k > rep->max_chi) rep->max_chi = k;
        // s_k and s_{k+1} equal to 1e-10 (their squares to 2e-10)
        if (k < r && k == p.chi_max && A::to_float(vnext) > 0.f &&
            fabsf(A::to_float(A::sub(vmin, vnext))) <= 2e-10f * A::to_float(vmin))
          rep->degenerate_cuts += 1;
        if (!converged) rep->not_converged += 1;
        const int used = converged ? sweep : p.max_sweeps + 1;
        if (used > rep->max_sweeps) rep->max_sweeps = used;
        rep->two_qubit_gates += 1;
        // nominal: a dot product (8 n) and a rotation (20 n) for every column pair
        // of every sweep, also where it was left out (counting the pairs that
        // were met and rotated took 2 to 3 % of a theta's time)
        rep->svd_flops += (double)(sweep * (r * (r - 1) / 2)) * (double)(28 * n);
        rep->sweeps_fp64 += sweep;
        rep->phase_cycles[0] += double(t_load - t_start);
        rep->phase_cycles[1] += double(t_gs - t_load);
        rep->phase_cycles[2] += double(t_sw - t_gs);
        rep->phase_cycles[3] += double(clock64() - t_sw);
        *chi_out = k;
      }
    }
  }
  // ---- B~_{q+1}[a, :] = conj(X[:, id]) / |X[:, id]|
  {
    const int items = nslots * b;
    const int lg = lanes_log2<A>(items, n), G = 1 << lg, gl = tid & (G - 1), grp = tid >> lg, NG = T >> lg;
    for (int i = grp; i < items; i += NG) {
      const int slot = i >= b ? 1 : 0, c = i - slot * b;
      const int blk = block_at(slot, 0), id = blk * b + c;
      if (id >= r || rnk[id] >= k) continue;
      const HX col = held(i, id);
      const S f = A::rsqrt(nA[id]);
      cplx<R>* out = Bnext + (size_t)rnk[id] * n;
      for (int rr = gl; rr < n; rr += G) {
        const V v = A::scale(A::template load<kGX>(col, ldx, rr), f);
        if constexpr (sizeof(R) == 8) {
          const double2 z = A::value(v);
          __stcg(out + rr, make_double2(z.x, -z.y));
        } else {
          const float2 z = A::value32(v);
          __stcg(out + rr, make_float2(z.x, -z.y));
        }
      }
    }
  }
  if (!refine) {
    __syncthreads();  // s_d[1]
    if (me == 0) {
      for (int id = tid; id < r; id += T)
        if (rnk[id] < k) lam_next[rnk[id]] = sqrt(sg[id]) * s_d[1];
      if (tid == 0) rep->inv_norm = s_d[1] * scl;
    }
    if (!Bq) return k;
  }
  const double w_unit = __longlong_as_double((long long)(1023 + max(-1000, min(1000, ec - ex))) << 52);
  S* kn = reinterpret_cast<S*>(nrm);  // squared kept values, in units of 4^ec
  // ||s||, and lam = s / ||s|| in descending order (a running minimum: the
  // refined values of a degenerate pair can differ in their last bits either
  // way), by warp 0.  Below 1e-18 of ||C|| (double-float: the FP32 range of the
  // roots' seeds) a value becomes a token, which keeps the direction alive for the
  // next gate on its bond.  FP64 sweeps are finished in FP64; the double-float
  // roots take one FP64 Newton step each.
  constexpr bool kF64 = std::is_same<A, ArF64>::value;
  auto finish_lam = [&](auto value) {
    if (tid < 32) {
      S kept = A::zero();
      for (int a = lane; a < k; a += 32) kept = A::add(kept, value(a));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) kept = A::shfl_add(kept, o);
      double inv;  // 1 / ||s|| in units of 2^-ec
      if constexpr (kF64) {
        inv = kept > 0.0 ? 1.0 / sqrt(kept) : 1.0;
      } else {
        const bool any = kept.h > 1e-36f;
        const double kd = any ? ff_join(kept) : 1.0;
        inv = ff_join(ff_rsqrt(any ? kept : ff_make(1.f, 0.f)));
        inv = inv * fma(-0.5 * kd * inv, inv, 1.5);
      }
      if (lane == 0) s_d[1] = inv;
      if (me == 0) {
        double run = 1e300;
        for (int a0 = 0; a0 < k; a0 += 32) {
          double l = run;
          if (a0 + lane < k) {
            const S v = value(a0 + lane);
            if constexpr (kF64) {
              l = v > 1e-36 ? sqrt(v) * inv : 1e-18;
            } else {
              const bool pos = v.h > 1e-36f;
              const double vd = pos ? ff_join(v) : 0.0, y = ff_join(ff_rsqrt(pos ? v : ff_make(1.f, 0.f)));
              const double s0 = vd * y;
              l = pos ? fma(0.5 * y, fma(-s0, s0, vd), s0) * inv : 1e-18;
            }
          }
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const double u = __shfl_up_sync(0xffffffffu, l, o);
            if (lane >= o && __double_as_longlong(u) < __double_as_longlong(l)) l = u;
          }
          if (__double_as_longlong(run) < __double_as_longlong(l)) l = run;
          run = __shfl_sync(0xffffffffu, l, 31);
          if (a0 + lane < k) lam_next[a0 + lane] = l;
        }
        if (lane == 0) {
          if (run < rep->min_kept_sv) rep->min_kept_sv = run;
          rep->inv_norm = inv * cscl;
        }
      }
    }
    __syncthreads();
  };

  cudaTriggerProgrammaticLaunchCompletion();  // the next gate's launch overlaps the rest
  if (direct) {
    // ---- one CTA: W = C V^H from shared memory, one column of W per group of
    // lanes (a lane takes every g-th row); W replaces A.  Against the tiles
    // below: no waits for L2 and no barriers inside, 17 -> 5 thousand cycles
    // at 16 x 16.
    int* order = reinterpret_cast<int*>(srt);
    for (int id = tid; id < r; id += T)
      if (rnk[id] < k) order[rnk[id]] = id;
    __syncthreads();
    int lg = 5;
    while (lg > 2 && (1 << (lg - 1)) >= m) --lg;
    const int g = 1 << lg, gl = tid & (g - 1), grp = tid >> lg, NG = T >> lg;
    for (int a0 = 0; a0 < k; a0 += NG) {
      const int a = a0 + grp;
      if (!__any_sync(0xffffffffu, a < k)) continue;
      const int id = order[min(a, k - 1)];
      const HX col = held(id, id);
      const S f = A::rsqrt(nA[id]);
      typename A::NAcc s2;
      for (int row = gl; row < m; row += g) {
        typename A::Acc acc;
#pragma unroll 2
        for (int c = 0; c < n; ++c)
          A::dot(acc, A::template load<false>(c0 + (unsigned)(c * ca), lda, row), A::template load<kGX>(col, ldx, c));
        S wr, wi;
        A::dot_sum(acc, 1, wr, wi);
        const V w = A::scale(A::cval(wr, wi), f);
        if (a < k) {
          if constexpr (!kGA) A::template store<false>(acol(a, a), lda, row, w);
          if (refine) A::nrm(s2, A::scale(w, A::from_double(__ldcg(lam_l + (row >> 1)))));
        }
      }
      S v = A::nrm_value(s2);
      for (int o = g >> 1; o > 0; o >>= 1) v = A::shfl_add(v, o);
      if (refine && a < k && gl == 0) kn[a] = v;
    }
    __syncthreads();
    if (refine)
      finish_lam([&](int a) { return kn[a]; });
    if (Bq) {
      const S inv = A::from_double(refine ? s_d[1] : s_d[1] * w_unit);
      for (int t = tid; t < m * k; t += T) {
        const int row = t / k, a = t - row * k;
        if constexpr (!kGA) {
          const V v = A::scale(A::template load<false>(acol(a, a), lda, row), inv);
          if constexpr (sizeof(R) == 8)
            Bq[t] = A::value(v);
          else
            Bq[t] = A::value32(v);
        }
      }
    }
    return k;
  }
  if (!tm.barrier()) return 0;  // every row of B~_{q+1} is written, X's shared memory is free

  // ---- W = C V^H
  using WA = A;  // complex64 states too: one rounding to FP32 instead of n
  using WV = typename WA::V;
  const unsigned sa = 0, sb = kPM * 20 * 16, sred = (kPM + kPK) * 20 * 16;
  constexpr int kLd = 20;                       // padded length of 16 entries (WA::ld(16) or more)
  constexpr unsigned kCol = kLd * WA::kBytes;   // bytes of a 16-entry run
  const int tx = tid & 15, ty = tid >> 4, TY = T >> 4, nrow = (kPM - ty + TY - 1) / TY;  // 2 to 4 rows a thread
  S* red = reinterpret_cast<S*>(svd_smem + sred);
  S* rowsq = reinterpret_cast<S*>(svd_smem + sa);  // of a tile's 64 rows, where C's tile was
  for (int j0 = me * kPN; j0 < k; j0 += P * kPN) {
    // sums of (lam |W|)^2 down a column: rows part, part + 16, ... by one thread
    // of the first 256, whatever the block size (a run's is another one)
    S col2 = A::zero();
    for (int r0 = 0; r0 < m; r0 += kPM) {
      typename WA::Acc acc[4];
      for (int c0 = 0; c0 < n; c0 += kPK) {
        for (int t = tid; t < kPM * kPK; t += T) {
          const int kk = t & 15, row = t >> 4;
          WV v = WA::zero_entry();
          if (r0 + row < m && c0 + kk < n) {
            const cplx<R> z = __ldcg(Cm + (size_t)(r0 + row) * n + c0 + kk);
            v = WA::make(z.x * cscl, z.y * cscl);
          }
          WA::template store<false>(sa + row * kCol, kLd, kk, v);
        }
        for (int t = tid; t < kPN * kPK; t += T) {
          const int kk = t & 15, j = t >> 4;
          WV v = WA::zero_entry();
          if (j0 + j < k && c0 + kk < n) {
            const cplx<R> z = __ldcg(Bnext + (size_t)(j0 + j) * n + c0 + kk);
            v = WA::make(z.x, z.y);
          }
          WA::template store<false>(sb + kk * kCol, kLd, j, v);
        }
        __syncthreads();
        const int kend = min(kPK, n - c0);
        for (int kk = 0; kk < kend; ++kk) {
          const WV bv = WA::template load<false>(sb + kk * kCol, kLd, tx);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (i < nrow && r0 + ty + i * TY < m)
              WA::dot(acc[i], bv, WA::template load<false>(sa + (ty + i * TY) * kCol, kLd, kk));
        }
        __syncthreads();
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int row = r0 + ty + i * TY;
        S sq = A::zero();
        if (i < nrow && row < m && j0 + tx < k) {
          typename WA::S wr, wi;
          WA::dot_sum(acc[i], 1, wr, wi);
          // W is in units of 2^ec, the norm in units of 2^ex; refine: scaled
          // below, when the norm is known
          if (Bq) {
            const double f = refine ? 1.0 : s_d[1] * w_unit;
            const double zr = WA::to_double(wr), zi = WA::to_double(wi);
            __stcg(Bq + (size_t)row * k + j0 + tx, refine ? cmk<R>(R(zr), R(zi)) : cmk<R>(R(zr * f), R(zi * f)));
          }
          if (refine) {
            const S w = A::from_double(__ldcg(lam_l + (row >> 1)));
            typename A::NAcc q2;
            A::nrm(q2, A::cval(A::mul(w, wr), A::mul(w, wi)));
            sq = A::nrm_value(q2);
          }
        }
        if (refine && i < nrow && ty + i * TY < kPM) rowsq[(ty + i * TY) * 16 + tx] = sq;
      }
      if (refine) {
        __syncthreads();
        if (tid < 256)
          for (int row = ty; row < kPM; row += 16) col2 = A::add(col2, rowsq[row * 16 + tx]);
        __syncthreads();
      }
    }
    if (refine) {
      if (tid < 256) {
        const S v1 = A::shfl_add(col2, 16);
        if (lane < 16) red[(tid >> 5) * 16 + tx] = v1;
      }
      __syncthreads();
      if (tid < 16 && j0 + tid < k) {
        S v = red[tid];
        for (int w = 1; w < 8; ++w) v = A::add(v, red[w * 16 + tid]);
        double d = 0.0;
        memcpy(&d, &v, sizeof(S));
        __stcg(gnrm + j0 + tid, d);
      }
      __syncthreads();
    }
  }
  if (refine) {
    if (!tm.barrier()) return 0;
    finish_lam([&](int a) {
      const double d = __ldcg(gnrm + a);
      S v;
      memcpy(&v, &d, sizeof(S));
      return v;
    });
  }
  // ---- scale this CTA's columns of B~_q (only it wrote and reads them)
  if (refine && Bq) {
    const S inv = A::from_double(s_d[1]);
    for (int j0 = me * kPN; j0 < k; j0 += P * kPN)
      for (int row = ty; row < m; row += TY)
        if (j0 + tx < k) {
          cplx<R>* z = Bq + (size_t)row * k + j0 + tx;
          const cplx<R> v = __ldcg(z);
          if constexpr (sizeof(R) == 8) *z = A::value(A::scale(A::make(v.x, v.y), inv));
        }
  }
  return k;
}

// ---- kernels ------------------------------------------------------------------
// (FP64 work is bound by the SM's two FP64 units, which a few warps fill.)
template <class A> constexpr int kSvdThreads = std::is_same<A, ArF64>::value ? 256 : 512;

// Columns up to which one CTA takes the theta although more were launched.
constexpr int kSvdSingleCols = 48;

// CTAs that a theta of m x n gets, by its sizes alone; 0: more than the Pl
// launched (a run's next tier or the grid kernel takes it).
template <class A>
__host__ __device__ inline int svd_team_size(int m, int n, int Pl) {
  if (n <= kSvdSingleCols && SvdSmem<A>::bytes(m, n, 1, true, true) <= kSvdSmemLimit) return 1;
  for (int P = 4; P <= Pl; P *= 2)
    if (SvdSmem<A>::bytes(m, n, P, true, true) <= kSvdSmemLimit) return P;
  return 0;
}

template <class A, class R>
__global__ void __launch_bounds__(kSvdThreads<A>, 1)
    svd_kernel(const cplx<R>* __restrict__ Cm, const double* __restrict__ lam_l, int* __restrict__ chi, int q,
               SvdParams p, cplx<R>* __restrict__ Bnext, double* __restrict__ lam_next, DevReport* __restrict__ rep,
               cplx<R>* __restrict__ Bq, char* __restrict__ gws) {
  __shared__ float2 s_mail[2 * 16];
  const int Pl = (int)cg::this_cluster().num_blocks(), me = (int)cg::this_cluster().block_rank();
  cudaGridDependencySynchronize();  // may be launched while the theta contraction runs
  const int m = 2 * __ldcg(chi + q), n = 2 * __ldcg(chi + q + 2);
  const int P = svd_team_size<A>(m, n, Pl);
  if (me >= P) return;  // an exited CTA counts as arrived at the cluster barriers
  if (P == 1) {
    OneTeam tm;
    svd_body<A, R, OneTeam, false>(tm, Cm, lam_l, m, n, p, Bnext, lam_next, chi + q + 1, rep, Bq, gws);
  } else {
    ClusterTeam tm{me, P, s_mail};
    tm.barrier();  // every CTA runs before its shared memory is written
    svd_body<A, R, ClusterTeam, false>(tm, Cm, lam_l, m, n, p, Bnext, lam_next, chi + q + 1, rep, Bq, gws);
  }
}

// Thetas that do not fit a cluster: a co-resident grid (cooperative launch).
// Pl: the CTAs of the cluster launch that ran before and may have done it.
template <class A, class R>
__global__ void __launch_bounds__(kSvdThreads<A>, 1)
    svd_grid_kernel(const cplx<R>* __restrict__ Cm, const double* __restrict__ lam_l, int* __restrict__ chi, int q,
                    SvdParams p, cplx<R>* __restrict__ Bnext, double* __restrict__ lam_next,
                    DevReport* __restrict__ rep, cplx<R>* __restrict__ Bq, char* __restrict__ gws, GridSync* sync, int Pl,
                    unsigned smem_bytes) {
  const int m = 2 * chi[q], n = 2 * chi[q + 2];
  if (svd_team_size<A>(m, n, Pl)) return;
  // a block of X needs at least one column on every CTA
  const int P = min((int)gridDim.x, max(2, (min(m, n) + 3) / 4));
  if ((int)blockIdx.x >= P) return;
  GridTeam tm{(int)blockIdx.x, P, sync, reinterpret_cast<float2*>(gws + SvdWs<A>(m, n, true).mail)};
  int k;
  if (SvdSmem<A>::bytes(m, n, P, false, true) <= smem_bytes)
    k = svd_body<A, R, GridTeam, false>(tm, Cm, lam_l, m, n, p, Bnext, lam_next, chi + q + 1, rep, Bq, gws);
  else
    k = svd_body<A, R, GridTeam, true>(tm, Cm, lam_l, m, n, p, Bnext, lam_next, chi + q + 1, rep, Bq, gws);
  if (k == 0 && threadIdx.x == 0) rep->tc_error = 1;  // any CTA that gave up: its part is missing
}

}  // namespace mpsv

// FP32 one-sided Jacobi SVD on a thread-block cluster (Algorithm 1 of the paper's
// "SVD and one-side jacobi" subsection, parallelised over up to 16 SMs).
//
// The kernel orthogonalises the n = 2 chi_r columns of A = C~ (m = 2 chi_l
// rows, read from the row-major theta C as A[r, c] = lam_q[r / 2] C[r, c])
// and accumulates the same rotations into V (Algorithm 1: A = A J, V = V J).
// Each column is stored as the stacked vector [A(:, c); V(:, c)] of length
// m + n, so one rotation updates both.  When the columns are orthogonal,
// A = U Sigma and V holds the right singular vectors W; the kept rows of
// B~_{q+1} = W^H are conjugated columns of V, unitary to rounding for any
// singular value (normalising columns of A instead would amplify the
// rounding error of small columns by s_1 / s_j).
//
// Parallel order.  The n columns are split into 2P blocks of b columns
// (zero-padded).  CTA p of the P-CTA cluster holds the blocks at positions p
// and 2P-1-p of a circle-method round robin over the 2P blocks: in each of
// the 2P-1 rounds of a sweep every CTA orthogonalises all column pairs
// between its two blocks (and, in the first round, also the pairs inside
// each block), then every block except the one at position 0 advances one
// position.  Blocks move through distributed shared memory into ping-pong
// buffers, so one cluster barrier per round orders the hand-over.  When the
// stacked columns do not fit the shared memory they stay in a global
// workspace, and a round only renames the positions.
//
// This form serves the FP32 SVD (mps_config.svd_fp64 = 0); the FP64-accurate
// SVDs run svd_jacobi.cuh.
#pragma once

#include <cooperative_groups.h>

#include "common.cuh"

namespace mpsv {

namespace cg = cooperative_groups;

// Rotation of a column pair of the one-sided Jacobi SVD from its Gram entries
// alpha = a_i^H a_i, beta = a_j^H a_j, g = gr + i gi = a_i^H a_j (Algorithm 1
// of the paper, with the phase of g moved onto column j): the new columns are
// a_i' = c a_i - conj(s e^{i phi}) a_j and a_j' = c a_j + s e^{i phi} a_i.
// Returns false when the pair is left alone: already orthogonal to tol, or a
// column at the rounding floor.
template <typename S>
__device__ __forceinline__ bool jacobi_rotation(S alpha, S beta, S gr, S gi, S tol, S floor, S tiny, S& c,
                                                cplx<S>& sph) {
  const S mag = sqrt(gr * gr + gi * gi);
  if (!(mag > tiny) || !(mag > tol * sqrt(alpha * beta)) || !(min(alpha, beta) > floor)) return false;
  const S zeta = (beta - alpha) / (S(2) * mag);
  const S t = (zeta >= S(0) ? S(1) : S(-1)) / (fabs(zeta) + sqrt(S(1) + zeta * zeta));
  c = S(1) / sqrt(S(1) + t * t);
  const S s = t * c;
  sph = cmk<S>(s * gr / mag, s * gi / mag);  // s e^{i phi}
  return true;
}

// The pair rules of the truncation SVD (tail columns).  Jacobi only has to
// make the columns that the truncation keeps orthogonal to each other and to
// all others; the columns it discards may stay mixed among themselves as long
// as none of their singular values could reach the cut.  At the start of a
// sweep, from the squared column norms nrm2[0..n): the kept set K is what the
// truncation would keep now (nrm2 > trunc_rel^2 max nrm2, the chi_max largest
// by rank when more pass), D the rest, and the cut is trunc_rel^2 max nrm2 (or
// the smallest kept nrm2 under a chi_max cut).  The class of column c goes to
// cls[c]:
//  * kTailSkip when sum_D nrm2 <= cut / 4: every singular value of the D
//    block is then at most half of every kept column's norm, so once K is
//    orthogonal to itself and to D, K holds the leading singular vectors
//    whatever D looks like (and the discarded weight is sum_D nrm2); pairs of
//    two such columns are not rotated.  The factor 1/4 also bounds how much
//    rotating a kept column against one D column disturbs its orthogonality
//    to the others, so the kept columns converge quickly (a bare per-column
//    threshold did not: a column just above it never converged against mixed
//    columns just below it).
//  * kTailLoose otherwise, for the deep tail T: the D columns with nrm2 <=
//    t_d, where t_d <= cut / 4 is the largest such norm below a gap, i.e.
//    the next larger nrm2 of any column is at least 4 t_d.  Pairs of two of
//    them are rotated only while |g| > loose_tol sqrt(b_ii b_jj), loose_tol =
//    min(2 / n, cut / (16 sum_T nrm2)), returned in *loose.  By Gershgorin on
//    their Gram matrix the singular values of T then stay below
//    (cut / 4)(1 + n loose_tol) < cut.  Every other column has nrm2 >= 4
//    t_d, so its rotations against T have small angles (|s| <= 4|g| / (3
//    nrm2)) and disturb its orthogonality to the rest of T by at most
//    loose_tol sum_T nrm2 / nrm2 <= 1/4 of what it was: it still converges.
//    (Without the gap a degenerate pair of columns straddling the threshold
//    rotated by large angles and carried the loose couplings of its deep
//    member into its tight one, and with 2 / n alone columns just above the
//    threshold crawled against many mixed columns just below it.)
//  * 0 for every other column (the normal stopping rule).
// Every thread of the block calls it; blocks with the same nrm2 and size
// compute the same classes.
constexpr int kTailLoose = 1, kTailSkip = 2;

__device__ __forceinline__ void truncation_tail(const double* nrm2, int n, double trunc_rel, int chi_max, int* cls,
                                                double* loose) {
  __shared__ double s_red[33];
  __shared__ int s_cnt;
  __shared__ double s_cut;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  // largest squared norm
  double mx = 0.0;
  for (int c = threadIdx.x; c < n; c += blockDim.x) mx = fmax(mx, nrm2[c]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) s_red[warp] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < nw; ++w) v = fmax(v, s_red[w]);
    s_red[32] = v;
    s_cnt = 0;
  }
  __syncthreads();
  const double thr = trunc_rel * trunc_rel * s_red[32];
  int cnt = 0;
  for (int c = threadIdx.x; c < n; c += blockDim.x) cnt += nrm2[c] > thr;
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if (lane == 0) atomicAdd(&s_cnt, cnt);
  __syncthreads();
  const bool by_rank = s_cnt > chi_max;
  if (threadIdx.x == 0) s_cut = thr;
  __syncthreads();
  // kept flags (1 = kept) into cls[] first
  for (int c = threadIdx.x; c < n; c += blockDim.x) {
    if (by_rank) {
      const double v = nrm2[c];
      int rk = 0;
      for (int h = 0; h < n; ++h) rk += (nrm2[h] > v) || (nrm2[h] == v && h < c);
      cls[c] = rk < chi_max;
      if (rk == chi_max - 1) s_cut = v;
    } else {
      cls[c] = nrm2[c] > thr;
    }
  }
  __syncthreads();
  // weight of D, summed in a fixed order
  double part = 0.0;
  for (int c = threadIdx.x; c < n; c += blockDim.x)
    if (!cls[c]) part += nrm2[c];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  __syncthreads();
  if (lane == 0) s_red[warp] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < nw; ++w) v += s_red[w];
    s_red[32] = v;
  }
  __syncthreads();
  const double cut = s_cut;
  const bool skip = s_red[32] <= 0.25 * cut;
  // deep-tail threshold t_d: the largest candidate norm (a discarded column
  // with nrm2 <= cut / 4) whose next larger norm among all columns is at
  // least 4 times it
  double td = -1.0;
  if (!skip)
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
      const double v = nrm2[c];
      if (cls[c] || !(v <= 0.25 * cut)) continue;
      double nxt = INFINITY;
      for (int h = 0; h < n; ++h)
        if (nrm2[h] > v) nxt = fmin(nxt, nrm2[h]);
      if (nxt >= 4.0 * v) td = fmax(td, v);
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) td = fmax(td, __shfl_xor_sync(0xffffffffu, td, o));
  __syncthreads();
  if (lane == 0) s_red[warp] = td;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = -1.0;
    for (int w = 0; w < nw; ++w) v = fmax(v, s_red[w]);
    s_red[32] = v;
  }
  __syncthreads();
  td = s_red[32];
  for (int c = threadIdx.x; c < n; c += blockDim.x)
    cls[c] = cls[c] ? 0 : (skip ? kTailSkip : (nrm2[c] <= td ? kTailLoose : 0));
  __syncthreads();
  // weight of the deep tail T, summed in a fixed order, for the loose tolerance
  part = 0.0;
  for (int c = threadIdx.x; c < n; c += blockDim.x)
    if (cls[c] == kTailLoose) part += nrm2[c];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  __syncthreads();
  if (lane == 0) s_red[warp] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < nw; ++w) v += s_red[w];
    const double l = 2.0 / n;
    *loose = v > 0.0 ? fmin(l, cut / (16.0 * v)) : l;
  }
  __syncthreads();
}

// The stopping tolerance of a pair from the classes of its columns (see
// truncation_tail): a negative value means the pair is not rotated.
template <typename S>
__device__ __forceinline__ S pair_tol(int ci, int cj, S tol, S loose) {
  const int c = min(ci, cj);
  return c == kTailSkip ? S(-1) : (c == kTailLoose ? max(tol, loose) : tol);
}

// Position (0 .. 2P-1) -> (CTA rank, slot 0 = top / 1 = bottom).
__device__ __forceinline__ void pos_owner(int pos, int P, int& rank, int& slot) {
  if (pos < P) {
    rank = pos;
    slot = 0;
  } else {
    rank = 2 * P - 1 - pos;
    slot = 1;
  }
}

// Stacked-column elements a lane keeps in registers in the cross rounds
// (columns up to 32 * kClusterRegs = 512 entries long).
constexpr int kClusterRegs = 16;

template <typename S>
__device__ __forceinline__ void warp_sum4(S& a, S& b, S& c, S& d) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
    c += __shfl_xor_sync(0xffffffffu, c, o);
    d += __shfl_xor_sync(0xffffffffu, d, o);
  }
}

// One warp rotates two stacked columns [A; V] held in shared memory; the Gram
// entries use the first m (A) rows.
template <typename S>
__device__ __forceinline__ int jacobi_pair_smem(cplx<S>* ai, cplx<S>* aj, int m, int len, int lane, S tol, S floor,
                                                S tiny) {
  using C = cplx<S>;
  S alpha = 0, beta = 0, gr = 0, gi = 0;
  for (int r = lane; r < m; r += 32) {
    const C x = ai[r], y = aj[r];
    alpha = fma(x.x, x.x, fma(x.y, x.y, alpha));
    beta = fma(y.x, y.x, fma(y.y, y.y, beta));
    gr = fma(x.x, y.x, fma(x.y, y.y, gr));
    gi = fma(x.x, y.y, fma(-x.y, y.x, gi));
  }
  warp_sum4(alpha, beta, gr, gi);
  S c;
  C sph;
  if (!jacobi_rotation(alpha, beta, gr, gi, tol, floor, tiny, c, sph)) return 0;
  for (int r = lane; r < len; r += 32) {
    const C x = ai[r], y = aj[r];
    ai[r] = csub(cmk<S>(c * x.x, c * x.y), cmulc(sph, y));
    aj[r] = cadd(cmk<S>(c * y.x, c * y.y), cmul(sph, x));
  }
  return 1;
}

// Same with the first column in registers: x[i] is row lane + 32 i.
template <typename S>
__device__ __forceinline__ int jacobi_pair_reg(cplx<S> (&x)[kClusterRegs], cplx<S>* aj, int m, int len, int lane,
                                               S tol, S floor, S tiny) {
  using C = cplx<S>;
  S alpha = 0, beta = 0, gr = 0, gi = 0;
#pragma unroll
  for (int i = 0; i < kClusterRegs; ++i) {
    const int r = lane + 32 * i;
    if (r < m) {
      const C xv = x[i], y = aj[r];
      alpha = fma(xv.x, xv.x, fma(xv.y, xv.y, alpha));
      beta = fma(y.x, y.x, fma(y.y, y.y, beta));
      gr = fma(xv.x, y.x, fma(xv.y, y.y, gr));
      gi = fma(xv.x, y.y, fma(-xv.y, y.x, gi));
    }
  }
  warp_sum4(alpha, beta, gr, gi);
  S c;
  C sph;
  if (!jacobi_rotation(alpha, beta, gr, gi, tol, floor, tiny, c, sph)) return 0;
#pragma unroll
  for (int i = 0; i < kClusterRegs; ++i) {
    const int r = lane + 32 * i;
    if (r < len) {
      const C xv = x[i], y = aj[r];
      x[i] = csub(cmk<S>(c * xv.x, c * xv.y), cmulc(sph, y));
      aj[r] = cadd(cmk<S>(c * y.x, c * y.y), cmul(sph, xv));
    }
  }
  return 1;
}



// |z|^2 of a stored column entry in double
template <typename C>
__device__ __forceinline__ double entry_nrm2(const C* col, int r) {
  return double(col[r].x) * col[r].x + double(col[r].y) * col[r].y;
}

// Cluster-uniform sizes of one SVD.
struct ClusterGeom {
  int Pl, me;   // CTAs launched, this CTA's rank
  int P, b;     // CTAs taking part, columns per block
  int m, ncols, len, ncols_pad;
  int nw, nt, wl, wp;
  bool member;  // me < P
};

// Column id (0 .. ncols_pad-1) of column c of the block in slot `slot` of
// CTA `me` in round `rnd` of a sweep: the block at position pos >= 1 has
// moved rnd places along the circle 1 .. 2P-1 since the sweep began, when
// position p held block p; position 0 keeps block 0.
__device__ __forceinline__ int col_id(const ClusterGeom& g, int slot, int c, int rnd) {
  const int pos = slot == 0 ? g.me : 2 * g.P - 1 - g.me;
  const int M = 2 * g.P - 1;
  const int blk = pos == 0 ? 0 : 1 + ((pos - 1 - rnd) % M + M) % M;
  return blk * g.b + c;
}

// Stacked columns of one precision: shared-memory ping-pong slots
// [pp][slot][c][len], or 2P global blocks [block][c][len] that stay put while
// the round robin renames positions.
// The layout is a template parameter so that the shared-memory form's
// pointers stay shared-memory pointers for the compiler (shared loads and
// stores rather than generic ones).
template <typename T, bool kGlobal>
struct ColStore {
  cplx<T>* base;  // shared-memory slots, or the global blocks
  int b, len, P, me;
  __device__ cplx<T>* col(int pp, int slot, int c, int rnd) const {
    if constexpr (!kGlobal) {
      return base + ((size_t)(pp * 2 + slot) * b + c) * len;
    } else {
      const int pos = slot == 0 ? me : 2 * P - 1 - me;
      const int M = 2 * P - 1;
      const int blk = pos == 0 ? 0 : 1 + ((pos - 1 - rnd) % M + M) % M;
      return base + ((size_t)blk * b + c) * len;
    }
  }
};

// Sweeps of the circle-method round robin: Jacobi rotations until a sweep
// rotates no pair (or max_sweeps).  Every CTA of the cluster calls it
// (non-members only keep the cluster barriers in step).  Returns the sweeps
// run.
//
// Tail rule: at the start of each sweep every CTA learns the squared norms of
// all columns (nrm2, through distributed shared memory) and marks the columns
// the truncation discards (truncation_tail, into tail[]); a pair of two
// marked columns is not rotated.
//
// Clean pairs: a pair whose two columns have not changed since the pair was
// last tested at the tight tolerance, and found orthogonal, is orthogonal
// still; it is not tested again.  Byte flags per column id, kept identical in
// every member CTA: dirty[] (rotated in this sweep; a rotation sets both
// columns' flags in every member CTA through distributed shared memory,
// visible by the next round's cluster barrier), dirty_prev[] (rotated in the
// previous sweep) and tight_prev[] (tail class 0 in the previous sweep).  A
// pair is clean when both columns are tight now and were in the previous
// sweep, and neither was rotated in the previous sweep or so far in this one.
// The first sweep tests every pair.
template <typename T, bool kGlobal>
__device__ __forceinline__ int cluster_sweeps(const ClusterGeom& g, const ColStore<T, kGlobal>& cs, int& cur, int max_sweeps, T tol, T floor,
                              T tiny, double trunc_rel, int chi_max, double* nrm2, int* tail, unsigned char* flags,
                              bool& converged, const cg::cluster_group& cluster, int* s_flag_in, int* s_any) {
  using C = cplx<T>;
  // In the cross rounds, when every warp has one top-slot column, warp w
  // keeps it in registers for the b rotations it takes part in; only the
  // bottom-slot columns are re-read, so one barrier per sub-round orders
  // their hand-off.
  const bool cache_x = g.len <= 32 * kClusterRegs && g.b <= g.nw;
  __shared__ double s_loose;
  T loose = T(0);  // the tail rule's loose tolerance of the sweep (pair_tol)
  const bool active = g.member && g.wp < g.b;
  unsigned char* dirty = flags;
  unsigned char* dirty_prev = flags + g.ncols_pad;
  unsigned char* tight_prev = flags + 2 * g.ncols_pad;
  for (int id = threadIdx.x; id < g.ncols_pad; id += g.nt) {
    dirty[id] = 0;
    dirty_prev[id] = 1;
    tight_prev[id] = 0;
  }
  __syncthreads();
  // a pair (column ids i, j) that needs no test (see above)
  auto clean = [&](int i, int j) -> bool {
    return tail[i] == 0 && tail[j] == 0 && tight_prev[i] && tight_prev[j] && !(dirty_prev[i] | dirty_prev[j] |
                                                                               dirty[i] | dirty[j]);
  };
  // both columns rotated: flag them in every member CTA (lane 0 of the warp)
  auto mark = [&](int i, int j) {
    if (g.wl != 0) return;
    for (int r2 = 0; r2 < g.P; ++r2) {
      unsigned char* d = r2 == g.me ? dirty : cluster.map_shared_rank(dirty, r2);
      d[i] = 1;
      d[j] = 1;
    }
  };
  int sweep = 0;
  converged = false;
  for (; sweep < max_sweeps; ++sweep) {
    int rotated = 0;
    // squared norms of this CTA's columns (positions hold their own blocks
    // at the start of a sweep) to every member CTA
    for (int c = g.wp; g.member && c < 2 * g.b; c += g.nw) {
      const C* a = cs.col(cur, c / g.b, c % g.b, 0);
      double acc = 0.0;
      for (int r = g.wl; r < g.m; r += 32) acc += entry_nrm2(a, r);
      acc = warp_sum(acc);
      if (g.wl == 0) {
        const int id = col_id(g, c / g.b, c % g.b, 0);
        for (int r2 = 0; r2 < g.P; ++r2) *cluster.map_shared_rank(nrm2 + id, r2) = acc;
      }
    }
    cluster.sync();
    if (g.member) {
      truncation_tail(nrm2, g.ncols_pad, trunc_rel, chi_max, tail, &s_loose);
      loose = T(s_loose);
    }
    for (int rnd = 0; rnd < 2 * g.P - 1; ++rnd) {
      if (!g.member) {
        // not taking part: only the cluster barrier below
      } else if (rnd == 0) {
        // every pair among the CTA's 2b columns: round robin over 2b players
        const int mod = 2 * g.b - 1;
        for (int sr = 0; sr < 2 * g.b - 1; ++sr) {
          for (int pw = g.wp; pw < g.b; pw += g.nw) {
            int a0, a1;
            if (pw == 0) {
              a0 = mod;
              a1 = sr;
            } else {
              a0 = (sr + pw) % mod;
              a1 = (sr - pw + mod) % mod;
            }
            C* x = cs.col(cur, a0 / g.b, a0 % g.b, rnd);
            C* y = cs.col(cur, a1 / g.b, a1 % g.b, rnd);
            const int i0 = col_id(g, a0 / g.b, a0 % g.b, rnd), i1 = col_id(g, a1 / g.b, a1 % g.b, rnd);
            const T tl = pair_tol(tail[i0], tail[i1], tol, loose);
            if (tl >= T(0) && !clean(i0, i1)) {
              const int r = jacobi_pair_smem<T>(x, y, g.m, g.len, g.wl, tl, floor, tiny);
              if (r) mark(i0, i1);
              rotated |= r;
            }
          }
          __syncthreads();
        }
      } else {
        C xr[kClusterRegs];
        C* xcol = cs.col(cur, 0, active ? g.wp : 0, rnd);
        if (active && cache_x) {
#pragma unroll
          for (int i = 0; i < kClusterRegs; ++i) {
            const int r = g.wl + 32 * i;
            xr[i] = r < g.len ? xcol[r] : cmk<T>(0, 0);
          }
        }
        for (int sr = 0; sr < g.b; ++sr) {
          if (cache_x) {
            if (active) {
              const int i0 = col_id(g, 0, g.wp, rnd), i1 = col_id(g, 1, (g.wp + sr) % g.b, rnd);
              const T tl = pair_tol(tail[i0], tail[i1], tol, loose);
              if (tl >= T(0) && !clean(i0, i1)) {
                const int r = jacobi_pair_reg<T>(xr, cs.col(cur, 1, (g.wp + sr) % g.b, rnd), g.m, g.len, g.wl, tl,
                                                 floor, tiny);
                if (r) mark(i0, i1);
                rotated |= r;
              }
            }
          } else {
            for (int pw = g.wp; pw < g.b; pw += g.nw) {
              C* x = cs.col(cur, 0, pw, rnd);
              C* y = cs.col(cur, 1, (pw + sr) % g.b, rnd);
              const int i0 = col_id(g, 0, pw, rnd), i1 = col_id(g, 1, (pw + sr) % g.b, rnd);
              const T tl = pair_tol(tail[i0], tail[i1], tol, loose);
              if (tl >= T(0) && !clean(i0, i1)) {
                const int r = jacobi_pair_smem<T>(x, y, g.m, g.len, g.wl, tl, floor, tiny);
                if (r) mark(i0, i1);
                rotated |= r;
              }
            }
          }
          __syncthreads();
        }
        if (active && cache_x) {
#pragma unroll
          for (int i = 0; i < kClusterRegs; ++i) {
            const int r = g.wl + 32 * i;
            if (r < g.len) xcol[r] = xr[i];
          }
        }
        __syncthreads();
      }
      if (g.P == 1) continue;  // a single CTA keeps its blocks (and needs no cluster barrier)
      if constexpr (!kGlobal) {
        // hand the blocks on: position pos -> pos + 1 (pos >= 1), 2P-1 -> 1
        const int nxt = cur ^ 1;
        const size_t units = (size_t)g.b * g.len * sizeof(C) / sizeof(uint4);
        for (int slot = 0; slot < 2 && g.member; ++slot) {
          const int pos = slot == 0 ? g.me : 2 * g.P - 1 - g.me;
          const int npos = pos == 0 ? 0 : (pos == 2 * g.P - 1 ? 1 : pos + 1);
          int drank, dslot;
          pos_owner(npos, g.P, drank, dslot);
          const uint4* src = reinterpret_cast<const uint4*>(cs.col(cur, slot, 0, 0));
          uint4* dst = reinterpret_cast<uint4*>(cluster.map_shared_rank(cs.col(nxt, dslot, 0, 0), drank));
          for (size_t t = threadIdx.x; t < units; t += g.nt) dst[t] = src[t];
        }
        cluster.sync();
        cur = nxt;
      } else {
        cluster.sync();  // global columns: this round's writes before the next round's reads
      }
    }
    // ---- convergence: every CTA tells every CTA whether it rotated
    if (threadIdx.x == 0) *s_any = 0;
    __syncthreads();
    if (rotated) *s_any = 1;
    __syncthreads();
    if (threadIdx.x < g.Pl) {
      int* dst = cluster.map_shared_rank(s_flag_in, (int)threadIdx.x);
      dst[g.me] = *s_any;
    }
    cluster.sync();
    int any = 0;
    for (int r2 = 0; r2 < g.Pl; ++r2) any |= s_flag_in[r2];
    cluster.sync();  // all reads done before the next sweep's writes
    // roll the clean-pair flags (no CTA writes dirty[] again before the next
    // sweep's norm exchange barrier)
    for (int id = threadIdx.x; g.member && id < g.ncols_pad; id += g.nt) {
      dirty_prev[id] = dirty[id];
      dirty[id] = 0;
      tight_prev[id] = tail[id] == 0;
    }
    __syncthreads();
    if (!any) {
      converged = true;
      ++sweep;
      break;
    }
  }
  return sweep;
}

// Threads per CTA of the cluster SVD.
constexpr int kClusterMaxThreads = 512;

template <typename S>
struct ClusterSvdSmem {
  // layout of the dynamic shared memory (offsets in bytes); len = m + n
  size_t buf, red, sig, rank, flags;
  size_t total;
  __host__ __device__ static size_t align16(size_t x) { return (x + 15) & ~size_t(15); }
  __host__ __device__ ClusterSvdSmem(int b, int len, int ncols_pad, int nthreads) {
    buf = 0;
    size_t slots = 2ull * 2 * b * len * sizeof(cplx<S>);  // ping-pong x {top, bottom}
    red = align16(buf + slots);
    sig = align16(red + 4ull * (nthreads / 32 + 1) * sizeof(S) * 2);
    rank = align16(sig + (size_t)ncols_pad * sizeof(double));
    flags = align16(rank + (size_t)ncols_pad * sizeof(int));  // three byte flags per column
    total = align16(flags + 3 * (size_t)ncols_pad) + 64;
  }
};

// Complex entries of the global workspace for a theta of capacity mcap x ncap:
// the stacked columns (at most 2 P - 1 padding columns, P <= 16).
__host__ __device__ inline size_t cluster_svd_workspace(size_t mcap, size_t ncap) {
  return (ncap + 32) * (mcap + ncap);
}

// Everything after the geometry: the column layout (shared or global) is a
// compile-time choice so that shared-memory accesses compile as such.
template <typename S, typename R, bool kGlobal>
__device__ __forceinline__ void svd_cluster_body(const ClusterGeom& g, const cg::cluster_group& cluster,
                                                 const cplx<R>* __restrict__ Cm, const double* __restrict__ lam_l,
                                                 int* __restrict__ chi, int q, const SvdParams& p,
                                                 cplx<R>* __restrict__ Bnext, double* __restrict__ lam_next,
                                                 DevReport* __restrict__ rep, cplx<S>* __restrict__ gbuf,
                                                 unsigned char* smem, int* s_flag_in, double* s_fro, int& s_k,
                                                 double& s_nrm, int* s_any, long long t_start) {
  using C = cplx<S>;
  const int m = g.m, ncols = g.ncols, len = g.len, b = g.b, P = g.P, me = g.me, nt = g.nt;
  const ClusterSvdSmem<S> L(b, kGlobal ? 0 : len, g.ncols_pad, nt);
  double* sig = reinterpret_cast<double*>(smem + L.sig);
  int* rnk = reinterpret_cast<int*>(smem + L.rank);
  const ColStore<S, kGlobal> cs{kGlobal ? gbuf : reinterpret_cast<C*>(smem + L.buf), b, len, P, me};

  // ---- load: position pos holds the initial block pos (columns pos*b ..)
  for (int slot = 0; slot < 2 && g.member; ++slot) {
    const int pos = slot == 0 ? me : 2 * P - 1 - me;
    for (size_t t = threadIdx.x; t < (size_t)b * len; t += nt) {
      const int c = (int)(t / len), r = (int)(t % len);
      const int col = pos * b + c;
      double vr = 0.0, vi = 0.0;
      if (col < ncols) {
        if (r < m) {
          const cplx<R> x = Cm[(size_t)r * ncols + col];
          const double w = lam_l[r >> 1];
          vr = w * double(x.x);
          vi = w * double(x.y);
        } else if (r - m == col) {
          vr = 1.0;
        }
      }
      cs.col(0, slot, c, 0)[r] = cmk<S>(S(vr), S(vi));
    }
  }
  // ||A||_F^2 from the theta: each CTA's share goes to every CTA, summed in rank order
  double part = 0.0;
  for (size_t t = threadIdx.x; g.member && t < (size_t)2 * b * m; t += nt) {
    const int c = (int)(t / m), r = (int)(t % m);
    const int pos = c < b ? me : 2 * P - 1 - me;
    const int col = pos * b + c % b;
    if (col >= ncols) continue;
    const cplx<R> x = Cm[(size_t)r * ncols + col];
    const double w = lam_l[r >> 1];
    part += w * w * (double(x.x) * x.x + double(x.y) * x.y);
  }
  part = warp_sum(part);
  if (threadIdx.x == 0) s_nrm = 0.0;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) atomicAdd(&s_nrm, part);
  __syncthreads();
  if (threadIdx.x < g.Pl) *cluster.map_shared_rank(&s_fro[me], (int)threadIdx.x) = s_nrm;
  cluster.sync();
  double fro2 = 0.0;
  for (int r2 = 0; r2 < g.Pl; ++r2) fro2 += s_fro[r2];

  // Stopping rule and rounding floor: rotate while |b_ij| > tol sqrt(b_ii b_jj)
  // with tol = 4 sqrt(max(m, n)) u (a few times the rounding error of a dot
  // product); columns with squared norm below (4 u ||A||_F)^2 are rounding
  // noise and left alone.
  const double tol_scale = 4.0 * sqrt(double(max(m, ncols)));
  // the tail rule's per-sweep scratch: squared norms and tail flags of all
  // columns (the singular values and ranks use the same arrays afterwards)
  double* nrm2 = sig;
  int* tail = rnk;
  unsigned char* flags = smem + L.flags;
  int cur = 0;
  bool converged = false;
  const long long t_load = clock64();
  const S eps_u = S(5.9604645e-08f);
  const S tol = p.tol > 0 ? S(p.tol) : S(tol_scale) * eps_u;
  const S floor = S(16.0 * double(eps_u) * double(eps_u) * fro2);
  const S tiny = S(1e-35f);
  const int sweep = cluster_sweeps<S, kGlobal>(g, cs, cur, p.max_sweeps, tol, floor, tiny, p.trunc_rel, p.chi_max, nrm2,
                                               tail, flags, converged, cluster, s_flag_in, s_any);

  // ---- singular values: norms of the A parts, shared with every CTA
  const int lane = g.wl, warp = g.wp;
  const int ncols_pad = g.ncols_pad;
  for (int c = warp; g.member && c < 2 * b; c += g.nw) {
    const C* a = cs.col(cur, c / b, c % b, 0);
    double acc = 0.0;
    for (int r = lane; r < m; r += 32) acc += entry_nrm2(a, r);
    acc = warp_sum(acc);
    if (lane == 0) {
      const double sv = sqrt(acc);
      const int gc = me * 2 * b + c;
      for (int r2 = 0; r2 < P; ++r2) *cluster.map_shared_rank(sig + gc, r2) = sv;
    }
  }
  cluster.sync();
  if (!g.member) {
    cluster.sync();  // pairs with the final barrier of the members
    return;
  }
  // ranks (descending, ties by index), the same in every CTA
  for (int gc = threadIdx.x; gc < ncols_pad; gc += nt) {
    const double sg = sig[gc];
    int rk = 0;
    for (int h = 0; h < ncols_pad; ++h) {
      const double sh = sig[h];
      rk += (sh > sg) || (sh == sg && h < gc);
    }
    rnk[gc] = rk;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double total = 0.0, smax = 0.0;
    for (int gc = 0; gc < ncols_pad; ++gc) {
      total += sig[gc] * sig[gc];
      smax = fmax(smax, sig[gc]);
    }
    int cnt = 0;
    for (int gc = 0; gc < ncols_pad; ++gc)
      if (p.trunc_rel > 0.0 ? (sig[gc] > p.trunc_rel * smax) : (sig[gc] > 0.0)) ++cnt;
    int k = min(cnt, min(p.chi_max, min(m, ncols)));
    if (k < 1) k = 1;
    double kept = 0.0, smin = 0.0, s_next = 0.0;
    for (int gc = 0; gc < ncols_pad; ++gc) {
      if (rnk[gc] < k) kept += sig[gc] * sig[gc];
      if (rnk[gc] == k - 1) smin = sig[gc];
      if (rnk[gc] == k) s_next = sig[gc];
    }
    double nrm = sqrt(kept);
    if (!(nrm > 0.0)) nrm = 1.0;
    s_k = k;
    s_nrm = nrm;
    if (me == 0) {
      rep->discarded_weight += total > 0.0 ? 1.0 - kept / total : 0.0;
      if (smin / nrm < rep->min_kept_sv) rep->min_kept_sv = smin / nrm;
      if (k > rep->max_chi) rep->max_chi = k;
      if (k < ncols && k == p.chi_max && s_next > 0.0 && fabs(smin - s_next) <= 1e-10 * smin)
        rep->degenerate_cuts += 1;
      if (!converged) rep->not_converged += 1;
      const int used_cap = converged ? sweep : p.max_sweeps + 1;
      if (used_cap > rep->max_sweeps) rep->max_sweeps = used_cap;
      rep->two_qubit_gates += 1;
      // per sweep and column pair: three dot products over m rows (16 m flops)
      // and one rotation of the stacked columns (12 (m + n) flops)
      rep->svd_flops += (double)sweep * 0.5 * ncols * (ncols - 1) * (16.0 * m + 12.0 * len);
      rep->inv_norm = 1.0 / nrm;
      rep->sweeps_fp32 += sweep;
      rep->phase_cycles[0] += double(t_load - t_start);
      rep->phase_cycles[2] += double(clock64() - t_load);
      chi[q + 1] = k;
    }
  }
  __syncthreads();
  const int k = s_k;
  const double inv = 1.0 / s_nrm;
  if (me == 0)
    for (int gc = threadIdx.x; gc < ncols_pad; gc += nt)
      if (rnk[gc] < k) lam_next[rnk[gc]] = sig[gc] * inv;
  // B~_{q+1}[a, :] = conj(V[:, gc]) for the column gc of rank a < k
  for (int c = warp; c < 2 * b; c += g.nw) {
    const int gc = me * 2 * b + c;
    const int a = rnk[gc];
    if (a >= k) continue;
    const C* v = cs.col(cur, c / b, c % b, 0) + m;
    for (int r = lane; r < ncols; r += 32) {
      Bnext[(size_t)a * ncols + r] = ccast<cplx<R>>(cconj(v[r]));
    }
  }
  cluster.sync();  // no CTA leaves while its shared memory may still be read
}


template <typename S, typename R>
__global__ void __launch_bounds__(kClusterMaxThreads, 1)
    svd_cluster_kernel(const cplx<R>* __restrict__ Cm, const double* __restrict__ lam_l, int* __restrict__ chi, int q,
                       SvdParams p, cplx<R>* __restrict__ Bnext, double* __restrict__ lam_next,
                       DevReport* __restrict__ rep, cplx<S>* __restrict__ gbuf, unsigned smem_bytes) {
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_flag_in[16];
  __shared__ double s_fro[16];
  __shared__ int s_k;
  __shared__ double s_nrm;
  __shared__ int s_any;

  const long long t_start = clock64();
  ClusterGeom g;
  g.Pl = (int)cluster.num_blocks();  // CTAs launched (sized for the bond capacities)
  g.me = (int)cluster.block_rank();
  const int chi_l = chi[q], chi_r = chi[q + 2];
  g.m = 2 * chi_l;      // rows of A
  g.ncols = 2 * chi_r;  // columns of A = rows of V
  g.len = g.m + g.ncols;
  g.nw = (int)(blockDim.x >> 5);
  g.nt = blockDim.x;
  g.wl = threadIdx.x & 31;
  g.wp = threadIdx.x >> 5;
  // CTAs that take part, from the actual bond dimensions: the pair steps are
  // latency-bound, so as few CTAs as the warps allow (fewer rounds and cluster
  // barriers).  The others (rank >= P) only keep the cluster barriers in step.
  const int per = g.nw;
  g.P = min(g.Pl, max(1, (g.ncols + 2 * per - 1) / (2 * per)));
  // Without a global workspace the columns must fit the launch's shared
  // memory: fewer CTAs mean wider blocks (an FP32 theta of 96 columns takes 3
  // CTAs of 16 columns where the capacity plan sized 4 of 12), so spread them
  // over more of the launched CTAs until they fit.  The plan guarantees that
  // all Pl CTAs fit the capacity, hence the actual sizes.
  while (gbuf == nullptr && g.P < g.Pl) {
    const int bb = (g.ncols + 2 * g.P - 1) / (2 * g.P);
    if (ClusterSvdSmem<S>(bb, g.len, 2 * g.P * bb, g.nt).total <= smem_bytes) break;
    ++g.P;
  }
  g.member = g.me < g.P;
  g.b = (g.ncols + 2 * g.P - 1) / (2 * g.P);  // a warp takes pairs w, w + nw, ...
  g.ncols_pad = 2 * g.P * g.b;

  // Shared memory when the stacked columns fit the launch's allocation, else the global workspace.
  const bool fits = ClusterSvdSmem<S>(g.b, g.len, g.ncols_pad, g.nt).total <= smem_bytes;
  if (!fits && gbuf == nullptr) {
    // unreachable for launches sized by the host plan; leave without touching
    // the state (every CTA returns before any cluster barrier) and report it
    // as a sweep-cap hit so that the caller sees MPS_ENOTCONV
    if (g.me == 0 && threadIdx.x == 0) atomicAdd(&rep->not_converged, 1);
    return;
  }
  const bool in_smem = fits;
  if (in_smem)
    svd_cluster_body<S, R, false>(g, cluster, Cm, lam_l, chi, q, p, Bnext, lam_next, rep, gbuf, smem, s_flag_in,
                                         s_fro, s_k, s_nrm, &s_any, t_start);
  else
    svd_cluster_body<S, R, true>(g, cluster, Cm, lam_l, chi, q, p, Bnext, lam_next, rep, gbuf, smem, s_flag_in,
                                        s_fro, s_k, s_nrm, &s_any, t_start);
}

// ---------------------------------------------------------------------------
// one CTA: thetas of fewer than 96 columns
// ---------------------------------------------------------------------------

// Round-robin (circle method) schedule: in round r of nn-1 rounds, pair k.
__device__ __forceinline__ void rr_pair(int r, int k, int nn, int& i, int& j) {
  const int mod = nn - 1;
  int a, b;
  if (k == 0) {
    a = mod;
    b = r;
  } else {
    a = (r + k) % mod;
    b = (r - k + mod) % mod;
  }
  i = min(a, b);
  j = max(a, b);
}

template <typename S> struct SvdEps;
template <> struct SvdEps<float> {
  static __device__ float unit() { return 5.9604645e-08f; }
  static __device__ float tiny() { return 1e-35f; }
};

// Jacobi sweeps on A (m x n, column-major) accumulating V (n x n, column-major).
// Returns the number of sweeps used (max_sweeps + 1 if not converged).
// Columns whose squared norm is at most `floor` (the rounding level of A)
// are left alone: rotating two of them only reshuffles rounding noise, and a
// rotation against a larger column would move it by less than that noise.
// Pairs of two columns the truncation discards follow the tail rules
// (truncation_tail, pair_tol); nrm2 and tail are n-entry shared-memory scratch.
template <typename S>
__device__ int jacobi_sweeps(cplx<S>* A, cplx<S>* V, int m, int n, int max_sweeps, S tol, S floor, double trunc_rel,
                             int chi_max, double* nrm2, int* tail, int* s_flag) {
  using C = cplx<S>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int nn = n + (n & 1);
  const int pairs = nn / 2;
  const S tiny = SvdEps<S>::tiny();
  int sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    for (int j = warp; j < n; j += nwarps) {
      double acc = 0.0;
      for (int row = lane; row < m; row += 32) {
        const C x = A[(size_t)j * m + row];
        acc += double(x.x) * x.x + double(x.y) * x.y;
      }
      acc = warp_sum(acc);
      if (lane == 0) nrm2[j] = acc;
    }
    __syncthreads();
    __shared__ double s_loose;
    truncation_tail(nrm2, n, trunc_rel, chi_max, tail, &s_loose);
    const S loose = S(s_loose);
    if (threadIdx.x == 0) *s_flag = 0;
    __syncthreads();
    bool rotated = false;
    for (int r = 0; r < nn - 1; ++r) {
      for (int k = warp; k < pairs; k += nwarps) {
        int i, j;
        rr_pair(r, k, nn, i, j);
        if (j >= n) continue;
        const S tl = pair_tol(tail[i], tail[j], tol, loose);
        if (tl < S(0)) continue;
        C* ai = A + (size_t)i * m;
        C* aj = A + (size_t)j * m;
        S alpha = 0, beta = 0;
        C gam = cmk<S>(0, 0);
        for (int row = lane; row < m; row += 32) {
          const C x = ai[row], y = aj[row];
          alpha = fma(x.x, x.x, fma(x.y, x.y, alpha));
          beta = fma(y.x, y.x, fma(y.y, y.y, beta));
          cfmac(gam, x, y);
        }
        alpha = warp_sum(alpha);
        beta = warp_sum(beta);
        gam.x = warp_sum(gam.x);
        gam.y = warp_sum(gam.y);
        S c;
        C sph;  // s e^{i phi}
        if (!jacobi_rotation<S>(alpha, beta, gam.x, gam.y, tl, floor, tiny, c, sph)) continue;
        rotated = true;
        for (int row = lane; row < m; row += 32) {
          const C x = ai[row], y = aj[row];
          C ni = cmk<S>(c * x.x, c * x.y);
          ni = csub(ni, cmulc(sph, y));  // - s e^{-i phi} y
          C nj = cmk<S>(c * y.x, c * y.y);
          nj = cadd(nj, cmul(sph, x));
          ai[row] = ni;
          aj[row] = nj;
        }
        C* vi = V + (size_t)i * n;
        C* vj = V + (size_t)j * n;
        for (int row = lane; row < n; row += 32) {
          const C x = vi[row], y = vj[row];
          C ni = cmk<S>(c * x.x, c * x.y);
          ni = csub(ni, cmulc(sph, y));
          C nj = cmk<S>(c * y.x, c * y.y);
          nj = cadd(nj, cmul(sph, x));
          vi[row] = ni;
          vj[row] = nj;
        }
      }
      __syncthreads();
    }
    if (lane == 0 && rotated) *s_flag = 1;
    __syncthreads();
    const int any = *s_flag;
    __syncthreads();
    if (!any) return sweep + 1;
  }
  return max_sweeps + 1;
}

// Dynamic shared memory: [A m*n | V n*n] (when use_smem) then sig[n] (double), perm[n] (int).
template <typename S, typename R>
__global__ void __launch_bounds__(1024, 1)
    svd_truncate_kernel(const cplx<R>* __restrict__ Cm, const double* __restrict__ lam_l, cplx<S>* __restrict__ Ag,
                        cplx<S>* __restrict__ Vg, int use_smem, int* __restrict__ chi, int q, SvdParams p,
                        cplx<R>* __restrict__ Bnext, double* __restrict__ lam_next, DevReport* __restrict__ rep) {
  using C = cplx<S>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_flag;
  __shared__ int s_k;
  __shared__ double s_nrm;
  const int chi_l = chi[q], chi_r = chi[q + 2];
  const int m = 2 * chi_l, n = 2 * chi_r;
  C* A = Ag;
  C* V = Vg;
  unsigned char* tail = smem_raw;
  if (use_smem) {
    A = reinterpret_cast<C*>(smem_raw);
    V = A + (size_t)m * n;
    tail = reinterpret_cast<unsigned char*>(V + (size_t)n * n);
  }
  // column-major A = lam C from the row-major theta
  for (size_t t = threadIdx.x; t < (size_t)m * n; t += blockDim.x) {
    const int col = (int)(t % n), row = (int)(t / n);
    const C o = ccast<C>(Cm[t]);
    const S lam = S(lam_l[row >> 1]);
    A[(size_t)col * m + row] = cmk<S>(lam * o.x, lam * o.y);
  }
  double* sig = reinterpret_cast<double*>(tail);
  int* perm = reinterpret_cast<int*>(sig + n);
  for (size_t t = threadIdx.x; t < (size_t)n * n; t += blockDim.x) {
    const size_t col = t / n, row = t % n;
    V[t] = cmk<S>(col == row ? S(1) : S(0), S(0));
  }
  __syncthreads();

  // rotate while |b_ij| > tol sqrt(b_ii b_jj), tol = 4 sqrt(max(m, n)) u
  const S tol = p.tol > 0 ? S(p.tol) : S(4.0 * sqrt(double(max(m, n)))) * SvdEps<S>::unit();
  // ||A||_F^2 sets the noise floor of a column
  {
    double part = 0.0;
    for (size_t t = threadIdx.x; t < (size_t)m * n; t += blockDim.x) {
      const double x = A[t].x, y = A[t].y;
      part += x * x + y * y;
    }
    part = warp_sum(part);
    if (threadIdx.x == 0) s_nrm = 0.0;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) atomicAdd(&s_nrm, part);
    __syncthreads();
  }
  const double fro2 = s_nrm;
  const S floor = S(16.0 * double(SvdEps<S>::unit()) * double(SvdEps<S>::unit()) * fro2);
  __syncthreads();
  const int sweeps = jacobi_sweeps<S>(A, V, m, n, p.max_sweeps, tol, floor, p.trunc_rel, p.chi_max, sig, perm, &s_flag);

  // sigma_j = ||A_j|| (Algorithm 1: column norms)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  for (int j = warp; j < n; j += nwarps) {
    double acc = 0.0;
    const C* aj = A + (size_t)j * m;
    for (int row = lane; row < m; row += 32) {
      const double x = aj[row].x, y = aj[row].y;
      acc += x * x + y * y;
    }
    acc = warp_sum(acc);
    if (lane == 0) sig[j] = sqrt(acc);
  }
  __syncthreads();
  // descending order, ties by index (deterministic)
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const double sj = sig[j];
    int rank = 0;
    for (int i = 0; i < n; ++i) {
      const double si = sig[i];
      rank += (si > sj) || (si == sj && i < j);
    }
    perm[rank] = j;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double total = 0.0;
    for (int a = 0; a < n; ++a) total += sig[perm[a]] * sig[perm[a]];
    const double smax = sig[perm[0]];
    int cnt = 0;
    for (int a = 0; a < n; ++a) {
      const double s = sig[perm[a]];
      if (p.trunc_rel > 0.0 ? (s > p.trunc_rel * smax) : (s > 0.0)) ++cnt;
    }
    int k = min(cnt, min(p.chi_max, min(m, n)));
    if (k < 1) k = 1;
    double kept = 0.0;
    for (int a = 0; a < k; ++a) kept += sig[perm[a]] * sig[perm[a]];
    double nrm = sqrt(kept);
    if (!(nrm > 0.0)) nrm = 1.0;
    s_k = k;
    s_nrm = nrm;
    rep->discarded_weight += total > 0.0 ? 1.0 - kept / total : 0.0;
    const double smin = sig[perm[k - 1]] / nrm;
    if (smin < rep->min_kept_sv) rep->min_kept_sv = smin;
    if (k > rep->max_chi) rep->max_chi = k;
    if (k < n && k == p.chi_max) {
      const double a0 = sig[perm[k - 1]], a1 = sig[perm[k]];
      if (a1 > 0.0 && fabs(a0 - a1) <= 1e-10 * a0) rep->degenerate_cuts += 1;
    }
    if (sweeps > p.max_sweeps) rep->not_converged += 1;
    if (sweeps > rep->max_sweeps) rep->max_sweeps = sweeps;
    rep->two_qubit_gates += 1;
    // per sweep and column pair: three dot products over m rows (16 m flops)
    // and one rotation of the A and V columns (12 (m + n) flops)
    rep->svd_flops += (double)min(sweeps, p.max_sweeps) * 0.5 * n * (n - 1) * (16.0 * m + 12.0 * (m + n));
    rep->sweeps_fp32 += min(sweeps, p.max_sweeps);
    rep->inv_norm = 1.0 / nrm;
    chi[q + 1] = k;
  }
  __syncthreads();
  const int k = s_k;
  const double inv = 1.0 / s_nrm;
  for (int a = threadIdx.x; a < k; a += blockDim.x) lam_next[a] = sig[perm[a]] * inv;
  // B~_{q+1}[a, c] = conj(V[c, perm[a]])   (V = W, right singular vectors)
  for (size_t t = threadIdx.x; t < (size_t)k * n; t += blockDim.x) {
    const int a = (int)(t / n), c = (int)(t % n);
    const C v = V[(size_t)perm[a] * n + c];
    Bnext[t] = ccast<cplx<R>>(cconj(v));
  }
}

}  // namespace mpsv

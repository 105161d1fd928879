// Pauli-sum energy kernels (arXiv:2303.03681, Eqs. expec1/expec2).
//
// <P> for a string with first non-identity site m and last n is
//   Tr( T_{P_n} ... T_{P_m}( diag(lam_m^2) ) ),
//   T_P(L)[b, d] = sum_{a, c, i} conj(B[a, i, b]) L[a, c] P[i, pi(i)] B[c, pi(i), d],
// where pi(i) is the column of the single nonzero entry of row i of the
// Pauli matrix.  Strings are arranged in a prefix trie; the environment L of
// a trie node is computed once and shared by every string through it.
//
// The prefixes go up to the middle of the chain only.  From the other end the
// suffixes run down to it, with
//   T*_P(R)[a, c] = sum conj(B[a, i, b]) P[i, pi(i)] B[c, pi(i), d] R[b, d]
// from the identity (the site tensors are right-canonical), and a string across
// the middle is <P> = sum_{bd} L[b, d] R[b, d].  The number of distinct
// prefixes of a molecular Hamiltonian grows with the cube of the sites they
// cover: meeting halfway takes 8.4 -> 3.4 ms for the 14,251 strings of 20 spin
// orbitals at chi = 64, and for the 571,876 of 50 it stores 176 thousand environments
// instead of 1.14 million.  T* is T with the site tensor transposed: the
// suffixes run on the same kernels over transposed copies, and what is written below for
// the left half holds for the right half with the bonds exchanged.
//
// Site j (level j) runs:
//   env_m_kernel      M^b_p = L_p B_j[:, b, :] for each parent entry p
//                     (L_p = diag(lam_j^2) for strings starting at j),
//   env_child_kernel  L_c = sum_i ph_i B_j[:, i, :]^H M^{pi(i)}_p for the
//                     nodes c under p that have children,
//   env_leaf_kernel   <P> = Re sum_i ph_i <B_j[:, i, :], M^{pi(i)}_p> for a
//                     string ending at j whose node has no children,
//   env_trace_kernel  <P> = Re Tr L_c for a string ending at a node with children
// (in the right half both weight the last bond with lam^2);
// env_cross_kernel sums the strings across the middle;
// energy_reduce_kernel sums c_k <P_k> in FP64 in a fixed order.
#pragma once

#include "common.cuh"
#include "gate_kernels.cuh"  // kTile, Mac
#include "internal.h"        // EnvGroup

namespace mpsv {

// (pi(0), pi(1), phase_0, phase_1) of I, X, Y, Z.
struct PauliRow {
  int p0, p1;
  double2 ph0, ph1;
};
__device__ __forceinline__ PauliRow pauli_row(int op) {
  PauliRow r;
  switch (op) {
    case 1:  // X
      r.p0 = 1; r.p1 = 0; r.ph0 = make_double2(1, 0); r.ph1 = make_double2(1, 0); break;
    case 2:  // Y = [[0,-i],[i,0]]
      r.p0 = 1; r.p1 = 0; r.ph0 = make_double2(0, -1); r.ph1 = make_double2(0, 1); break;
    case 3:  // Z
      r.p0 = 0; r.p1 = 1; r.ph0 = make_double2(1, 0); r.ph1 = make_double2(-1, 0); break;
    default:  // I
      r.p0 = 0; r.p1 = 1; r.ph0 = make_double2(1, 0); r.ph1 = make_double2(1, 0); break;
  }
  return r;
}

struct EnvLevel {
  const int* parent_src;  // per parent entry: slot in the previous environment buffer, -1 = diag(lam^2)
  const EnvGroup* group;  // per parent entry with materialised children
  const int4* leaf;       // per string ending at a leaf node: (parent entry, op, term, 0)
  const int2* trace;      // per string ending at a materialised node: (slot, term)
  int n_parents, n_groups, n_leaves, n_traces;
  int chi_l, chi_r;        // bond dimensions the step comes from and goes to
  const double* weight;    // lam of the bond that leaves and traces end on (null: ones)
};

// M_p[a][b][d] = sum_c L_p[a][c] B[c][b][d]   (b = 0, 1): row-major chi_l x 2 chi_r,
// i.e. M_p = L_p B with B viewed as chi_l x 2 chi_r; slot stride of M: 2 chi_l chi_r
template <typename R>
__global__ void __launch_bounds__(kTile* kTile)
    env_m_kernel(const cplx<R>* __restrict__ Lprev, const cplx<R>* __restrict__ B, const double* __restrict__ lam,
                 EnvLevel lv, cplx<R>* __restrict__ M) {
  using C = cplx<R>;
  const int chi_l = lv.chi_l, chi_r = lv.chi_r;
  const int tiles_c = (lv.chi_r + kTile - 1) / kTile, tiles_r = (lv.chi_l + kTile - 1) / kTile;
  const int per = tiles_c * tiles_r;
  const int p = blockIdx.x / per, tile = blockIdx.x % per;
  const int a0 = (tile / tiles_c) * kTile, d0 = (tile % tiles_c) * kTile;
  if (p >= lv.n_parents || a0 >= chi_l || d0 >= chi_r) return;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int src = lv.parent_src[p];
  C* out = M + (size_t)p * 2 * lv.chi_l * lv.chi_r;
  const int a = a0 + ty, d = d0 + tx;
  const C zero = cmk<R>(0, 0);
  if (src < 0) {
    if (a < chi_l && d < chi_r) {
      const R w = lam ? R(lam[a] * lam[a]) : R(1);
      const C b0 = B[(size_t)(a * 2 + 0) * chi_r + d], b1 = B[(size_t)(a * 2 + 1) * chi_r + d];
      out[(size_t)a * 2 * chi_r + d] = cscale(b0, w);
      out[(size_t)a * 2 * chi_r + chi_r + d] = cscale(b1, w);
    }
    return;
  }
  using MT = Mac<R>;
  using E = typename MT::Elem;
  const C* L = Lprev + (size_t)src * lv.chi_l * lv.chi_l;
  __shared__ E sL[kTile][kTile + 1];
  __shared__ E sB[2][kTile][kTile + 1];
  typename MT::Acc acc0, acc1;
  for (int c0 = 0; c0 < chi_l; c0 += kTile) {
    sL[ty][tx] = (a < chi_l && c0 + tx < chi_l) ? MT::load(L[(size_t)a * chi_l + c0 + tx]) : MT::zero();
    const int c = c0 + ty;
    const bool ok = c < chi_l && d < chi_r;
    sB[0][ty][tx] = ok ? MT::load(B[(size_t)(c * 2 + 0) * chi_r + d]) : MT::zero();
    sB[1][ty][tx] = ok ? MT::load(B[(size_t)(c * 2 + 1) * chi_r + d]) : MT::zero();
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < kTile; ++kk) {
      const E l = sL[ty][kk];
      MT::fma(acc0, l, sB[0][kk][tx]);
      MT::fma(acc1, l, sB[1][kk][tx]);
    }
    __syncthreads();
  }
  if (a < chi_l && d < chi_r) {
    out[(size_t)a * 2 * chi_r + d] = MT::value(acc0);
    out[(size_t)a * 2 * chi_r + chi_r + d] = MT::value(acc1);
  }
}

// L_c[b][d] = sum_i ph_i sum_a conj(B[a][i][b]) M^{pi(i)}_p[a][d] for every child
// c of a parent p: with S_ij = B_i^H M_j
//   L_I = S_00 + S_11,  L_Z = S_00 - S_11,  L_X = S_01 + S_10,  L_Y = -i S_01 + i S_10.
// The four share the S_ij, and each is Hermitian (diag(lam^2) is, and a Pauli
// matrix keeps it so): a block takes one 16 x 16 tile on or above the diagonal,
// all children of its parent, and writes the mirrored tile too.  FP32
// arithmetic bounds it (double-float for complex128): 4.8 ms -> 3.6 ms for the
// 14,251 strings of 10 orbitals at chi = 64, against one child and every tile.
template <typename R>
__global__ void __launch_bounds__(kTile* kTile)
    env_child_kernel(const cplx<R>* __restrict__ M, const cplx<R>* __restrict__ B, EnvLevel lv,
                     cplx<R>* __restrict__ Lcur) {
  using C = cplx<R>;
  const int chi_l = lv.chi_l, chi_r = lv.chi_r;
  const int tiles = (lv.chi_r + kTile - 1) / kTile;
  const int per = tiles * (tiles + 1) / 2;
  const int gidx = blockIdx.x / per;
  int bi = 0, di = blockIdx.x % per;  // the tile's row and, counted from the diagonal, column
  while (di >= tiles - bi) di -= tiles - bi++;
  const int b0 = bi * kTile, d0 = (bi + di) * kTile;
  if (gidx >= lv.n_groups || d0 >= chi_r) return;
  const EnvGroup gr = lv.group[gidx];
  const bool iz = gr.slot[0] >= 0 || gr.slot[3] >= 0, xy = gr.slot[1] >= 0 || gr.slot[2] >= 0;
  const C* M0 = M + (size_t)gr.parent * 2 * lv.chi_l * lv.chi_r;  // row stride 2 chi_r
  const C* M1 = M0 + chi_r;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int b = b0 + ty, d = d0 + tx;
  using MT = Mac<R>;
  using E = typename MT::Elem;
  __shared__ E sB[2][kTile][kTile + 1];  // [i][a][b]
  __shared__ E sM[2][kTile][kTile + 1];  // [i][a][d]
  typename MT::Acc s00, s11, s01, s10;
  for (int a0 = 0; a0 < chi_l; a0 += kTile) {
    const int a = a0 + ty;
    const int bb = b0 + tx;
    const bool okb = a < chi_l && bb < chi_r;
    sB[0][ty][tx] = okb ? MT::load(B[(size_t)(a * 2 + 0) * chi_r + bb]) : MT::zero();
    sB[1][ty][tx] = okb ? MT::load(B[(size_t)(a * 2 + 1) * chi_r + bb]) : MT::zero();
    const bool okm = a < chi_l && d < chi_r;
    sM[0][ty][tx] = okm ? MT::load(M0[(size_t)a * 2 * chi_r + d]) : MT::zero();
    sM[1][ty][tx] = okm ? MT::load(M1[(size_t)a * 2 * chi_r + d]) : MT::zero();
    __syncthreads();
    const int kend = min(kTile, chi_l - a0);
    if (iz && xy) {
#pragma unroll 2
      for (int kk = 0; kk < kend; ++kk) {
        const E x0 = sB[0][kk][ty], x1 = sB[1][kk][ty], y0 = sM[0][kk][tx], y1 = sM[1][kk][tx];
        MT::fmac(s00, x0, y0);
        MT::fmac(s11, x1, y1);
        MT::fmac(s01, x0, y1);
        MT::fmac(s10, x1, y0);
      }
    } else if (iz) {
#pragma unroll 4
      for (int kk = 0; kk < kend; ++kk) {
        MT::fmac(s00, sB[0][kk][ty], sM[0][kk][tx]);
        MT::fmac(s11, sB[1][kk][ty], sM[1][kk][tx]);
      }
    } else {
#pragma unroll 4
      for (int kk = 0; kk < kend; ++kk) {
        MT::fmac(s01, sB[0][kk][ty], sM[1][kk][tx]);
        MT::fmac(s10, sB[1][kk][ty], sM[0][kk][tx]);
      }
    }
    __syncthreads();
  }
  if (d >= chi_r || b > d) return;
  const C p = MT::value_conj(s00), q = MT::value_conj(s11);
  const C u = MT::value_conj(s01), v = MT::value_conj(s10);
  const size_t size = (size_t)lv.chi_r * lv.chi_r;
  auto put = [&](int slot, C z) {
    if (slot < 0) return;
    C* out = Lcur + slot * size;
    out[(size_t)b * chi_r + d] = z;
    if (b != d) out[(size_t)d * chi_r + b] = cmk<R>(z.x, -z.y);
  };
  put(gr.slot[0], cadd(p, q));
  put(gr.slot[3], cmk<R>(p.x - q.x, p.y - q.y));
  put(gr.slot[1], cadd(u, v));
  put(gr.slot[2], cmk<R>(u.y - v.y, v.x - u.x));  // -i u + i v
}

// Sums of real products for string values: FP64 for complex128 states (splitting
// their entries costs more than the FP64 multiply-adds: the 14,251 strings of 10
// orbitals at chi = 64 take 3.40 ms, in double-float 3.56), and double-float for
// complex64 ones, whose entries' products are exact in it.
template <typename R> struct RealSum;
template <> struct RealSum<double> {
  using E = double;
  double v = 0.0;
  static __device__ __forceinline__ E elem(double x) { return x; }
  static __device__ __forceinline__ E mul(E a, E b) { return a * b; }
  __device__ __forceinline__ void add(E a, E b) { v = fma(a, b, v); }
  __device__ __forceinline__ E over_warp() const { return warp_sum(v); }
  static __device__ __forceinline__ double join(E a, E b, E c, E d) { return (a + b) + (c + d); }
};
template <> struct RealSum<float> {
  using E = ff;
  GramAcc v;
  static __device__ __forceinline__ E elem(float x) { return ff_make(x, 0.f); }
  static __device__ __forceinline__ E elem(double x) { return ff_split(x); }
  static __device__ __forceinline__ E mul(E a, E b) { return ff_mul(a, b); }
  __device__ __forceinline__ void add(E a, E b) { v.add(a, b); }
  __device__ __forceinline__ E over_warp() const {
    ff s = v.value();
    for (int x = 16; x > 0; x >>= 1) s = ff_add(s, ff_shfl_xor(s, x));
    return s;
  }
  static __device__ __forceinline__ double join(E a, E b, E c, E d) { return ff_join(ff_add(ff_add(a, b), ff_add(c, d))); }
};

// One block of four warps per leaf: Re sum_i ph_i sum_{a,b} conj(B[a][i][b]) M^{pi(i)}[a][b].
// One warp per leaf was a chain of 128 iterations at chi = 64: 0.8 of 8.4 ms for
// the strings of 10 orbitals.
template <typename R>
__global__ void __launch_bounds__(128)
    env_leaf_kernel(const cplx<R>* __restrict__ M, const cplx<R>* __restrict__ B, EnvLevel lv,
                    double* __restrict__ vals) {
  using C = cplx<R>;
  const int tid = threadIdx.x;
  const int chi_l = lv.chi_l, chi_r = lv.chi_r;
  const int4 lf = lv.leaf[blockIdx.x];
  const PauliRow pr = pauli_row(lf.y);
  const C ph0 = ccast<C>(pr.ph0), ph1 = ccast<C>(pr.ph1);
  const C* Mp = M + (size_t)lf.x * 2 * lv.chi_l * lv.chi_r;
  const C* Mi0 = Mp + (size_t)pr.p0 * chi_r;  // row stride 2 chi_r
  const C* Mi1 = Mp + (size_t)pr.p1 * chi_r;
  using Sum = RealSum<R>;
  Sum acc;
  const int tot = chi_l * chi_r;
#pragma unroll 2
  for (int t = tid; t < tot; t += 128) {
    const int a = t / chi_r, b = t - a * chi_r;
    const size_t at = (size_t)a * 2 * chi_r + b;
    const C x0 = B[at], x1 = B[at + chi_r];
    const C y0 = cmul(ph0, Mi0[at]), y1 = cmul(ph1, Mi1[at]);  // phases of 1, -1, i, -i: exact
    typename Sum::E f0 = Sum::elem(x0.x), f1 = Sum::elem(x0.y), f2 = Sum::elem(x1.x), f3 = Sum::elem(x1.y);
    if (lv.weight) {
      typename Sum::E w = Sum::elem(lv.weight[b]);
      w = Sum::mul(w, w);
      f0 = Sum::mul(w, f0);
      f1 = Sum::mul(w, f1);
      f2 = Sum::mul(w, f2);
      f3 = Sum::mul(w, f3);
    }
    acc.add(f0, Sum::elem(y0.x));
    acc.add(f1, Sum::elem(y0.y));
    acc.add(f2, Sum::elem(y1.x));
    acc.add(f3, Sum::elem(y1.y));
  }
  __shared__ typename Sum::E part[4];
  const typename Sum::E s = acc.over_warp();
  if ((tid & 31) == 0) part[tid >> 5] = s;
  __syncthreads();
  if (tid == 0) vals[lf.z] = Sum::join(part[0], part[1], part[2], part[3]);
}

// One warp per string ending at a materialised node: Re Tr L.
template <typename R>
__global__ void env_trace_kernel(const cplx<R>* __restrict__ Lcur, EnvLevel lv, double* __restrict__ vals) {
  const int lane = threadIdx.x & 31;
  const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (w >= lv.n_traces) return;
  const int chi_r = lv.chi_r;
  const int2 tr = lv.trace[w];
  const cplx<R>* L = Lcur + (size_t)tr.x * lv.chi_r * lv.chi_r;
  double s = 0.0;
  for (int b = lane; b < chi_r; b += 32) {
    const double wt = lv.weight ? lv.weight[b] * lv.weight[b] : 1.0;
    s += wt * (double)L[(size_t)b * chi_r + b].x;
  }
  s = warp_sum(s);
  if (lane == 0) vals[tr.y] = s;
}

// Transposed site tensors of the right half, [d][i][a] from [a][i][d], one after
// another (blockIdx.y: the site).
template <typename R>
__global__ void transpose_sites_kernel(const cplx<R>* __restrict__ B, const size_t* __restrict__ site_off,
                                       const int* __restrict__ chi, int cut, cplx<R>* __restrict__ BT) {
  const int site = cut + blockIdx.y, cl = chi[site], cr = chi[site + 1];
  size_t off = 0;
  for (int s = cut; s < site; ++s) off += (size_t)2 * chi[s] * chi[s + 1];
  const cplx<R>* src = B + site_off[site];
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < 2 * cl * cr; t += gridDim.x * blockDim.x) {
    const int d = t / (2 * cl), e = t - d * 2 * cl, i = e >= cl, a = e - i * cl;
    BT[off + t] = src[(size_t)(a * 2 + i) * cr + d];
  }
}

// <P> = sum_{bd} L[b][d] R[b][d] of the strings across the middle: both are
// Hermitian, so it is the sum over d >= b of Re(L R), twice off the diagonal.
// One block of four warps takes up to kCross strings of one prefix, so L is
// read once for them and the loads of the R (L2 latency bounds it) are in flight together;
// a group's missing strings repeat its last one.  Row p of the triangle is joined
// to row chi - 1 - p, which gives chi + 1 entries.
constexpr int kCross = 8;
template <typename R>
__global__ void __launch_bounds__(128)
    env_cross_kernel(const cplx<R>* __restrict__ L, const cplx<R>* __restrict__ Rm, int chi,
                     const int4* __restrict__ item, const int2* __restrict__ pair, double* __restrict__ vals) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int4 it = item[blockIdx.x];
  const size_t size = (size_t)chi * chi;
  const cplx<R>* Lp = L + it.x * size;
  const cplx<R>* Rp[kCross];
  using Sum = RealSum<R>;
  Sum acc[kCross];
#pragma unroll
  for (int k = 0; k < kCross; ++k) Rp[k] = Rm + pair[it.y + min(k, it.z - 1)].x * size;
  const int total = chi * (chi + 1) / 2;
  int p = 0, o = tid;
  for (int t = tid; t < total; t += 128, o += 128) {
    while (o > chi) {
      o -= chi + 1;
      ++p;
    }
    const int b = o < chi - p ? p : chi - 1 - p, d = o < chi - p ? p + o : o - 1;
    const size_t at = (size_t)b * chi + d;
    const cplx<R> z = Lp[at];
    cplx<R> v[kCross];
#pragma unroll
    for (int k = 0; k < kCross; ++k) v[k] = Rp[k][at];
    const R f = b == d ? R(1) : R(2);
    const typename Sum::E zr = Sum::elem(f * z.x), zi = Sum::elem(-f * z.y);
#pragma unroll
    for (int k = 0; k < kCross; ++k) {
      acc[k].add(zr, Sum::elem(v[k].x));
      acc[k].add(zi, Sum::elem(v[k].y));
    }
  }
  __shared__ typename Sum::E part[4][kCross];
#pragma unroll
  for (int k = 0; k < kCross; ++k) {
    const typename Sum::E s = acc[k].over_warp();
    if (lane == k) part[tid >> 5][k] = s;
  }
  __syncthreads();
  if (tid < it.z)
    vals[pair[it.y + tid].y] = Sum::join(part[0][tid], part[1][tid], part[2][tid], part[3][tid]);
}

// E = constant + sum_k c_k vals[k] (terms with an empty support keep vals = 1).
// One block of 1024 threads; fixed summation order.
// A set *err (a bounded wait of this state's kernels ran out) turns the energy into NaN.
static __global__ void energy_reduce_kernel(const double* __restrict__ vals, const double* __restrict__ coeffs,
                                            long long n_terms, double constant, const int* __restrict__ err,
                                            double* __restrict__ out) {
  __shared__ double part[32];
  double s = 0.0;
  for (long long k = threadIdx.x; k < n_terms; k += blockDim.x) s += coeffs[k] * vals[k];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.0;
    v = warp_sum(v);
    if (threadIdx.x == 0) *out = (err && *err) ? __longlong_as_double(0x7ff8000000000000ll) : constant + v;
  }
}

static __global__ void fill_kernel(double* __restrict__ p, long long n, double v) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) p[t] = v;
}

// Linear observables of the per-string values (reduced density matrices):
// out[r] = sum_{e in [row_ptr[r], row_ptr[r+1])} w[e] * vals[cols[e]], complex
// weights, FP64.  One warp per row; lane l takes the entries l, l + 32, ...
// and the lanes are summed in a fixed tree, so the result does not depend on
// the launch.  blockDim.x must be a multiple of 32 (whole warps leave
// together, so the shuffles see full warps).
static __global__ void observables_kernel(const double* __restrict__ vals, const long long* __restrict__ row_ptr,
                                          const int* __restrict__ cols, const double2* __restrict__ w,
                                          long long n_rows, double2* __restrict__ out) {
  const long long r = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (r >= n_rows) return;
  double re = 0.0, im = 0.0;
  const long long end = row_ptr[r + 1];
  for (long long e = row_ptr[r] + lane; e < end; e += 32) {
    const double v = vals[cols[e]];
    const double2 c = w[e];
    re = fma(c.x, v, re);
    im = fma(c.y, v, im);
  }
  re = warp_sum(re);
  im = warp_sum(im);
  if (lane == 0) out[r] = make_double2(re, im);
}

// ---------------------------------------------------------------------------
// tensor-core forms (complex64 states): the same products as env_m_kernel and
// env_child_kernel, as problems of tc::cgemm_kernel
// ---------------------------------------------------------------------------

// M_p = L_src B_j for the parents whose environment is a stored matrix;
// list[z] = (parent entry p, environment slot src).
struct EnvMProb {
  const int2* list;
  const float2* Lprev;
  const float2* B;
  float2* M;
  int chi_l, chi_r;
  __device__ __forceinline__ void dims(int, int& m, int& n, int& k) const {
    m = chi_l;
    n = 2 * chi_r;
    k = chi_l;
  }
  __device__ __forceinline__ float2 a(int z, int row, int kk) const {
    return Lprev[(size_t)list[z].y * chi_l * chi_l + (size_t)row * chi_l + kk];
  }
  __device__ __forceinline__ float2 b(int, int kk, int col) const { return B[(size_t)kk * 2 * chi_r + col]; }
  __device__ __forceinline__ void store(int z, int row, int col, float2 v) const {
    M[(size_t)list[z].x * 2 * chi_l * chi_r + (size_t)row * 2 * chi_r + col] = v;
  }
};

// L_c[b][d] = sum_{i, a} ph_i conj(B[a][i][b]) M_p[a][pi(i)][d]; K runs over (i, a).
struct EnvChildProb {
  const int2* child;  // (parent entry, op)
  const float2* B;
  const float2* M;
  float2* Lcur;
  int chi_l, chi_r;
  __device__ __forceinline__ void dims(int, int& m, int& n, int& k) const {
    m = chi_r;
    n = chi_r;
    k = 2 * chi_l;
  }
  __device__ __forceinline__ float2 a(int z, int row, int kk) const {
    const int i = kk >= chi_l ? 1 : 0, aa = kk - i * chi_l;
    const PauliRow pr = pauli_row(child[z].y);
    const double2 ph = i ? pr.ph1 : pr.ph0;
    const float2 x = B[(size_t)(aa * 2 + i) * chi_r + row];  // conj(x) * ph
    return make_float2(float(ph.x) * x.x + float(ph.y) * x.y, float(ph.y) * x.x - float(ph.x) * x.y);
  }
  __device__ __forceinline__ float2 b(int z, int kk, int col) const {
    const int i = kk >= chi_l ? 1 : 0, aa = kk - i * chi_l;
    const int2 cd = child[z];
    const PauliRow pr = pauli_row(cd.y);
    const int pi = i ? pr.p1 : pr.p0;
    return M[(size_t)cd.x * 2 * chi_l * chi_r + (size_t)aa * 2 * chi_r + (size_t)pi * chi_r + col];
  }
  __device__ __forceinline__ void store(int z, int row, int col, float2 v) const {
    Lcur[(size_t)z * chi_r * chi_r + (size_t)row * chi_r + col] = v;
  }
};

// M_p = diag(lam^2) B for the parents that start strings at this site; list[z] = entry p.
template <typename R>
__global__ void env_m_diag_kernel(const int* __restrict__ list, int n, const cplx<R>* __restrict__ B,
                                  const double* __restrict__ lam, int chi_l, int chi_r, cplx<R>* __restrict__ M) {
  const size_t per = (size_t)chi_l * 2 * chi_r;
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= per * n) return;
  const int z = (int)(t / per);
  const size_t e = t % per;
  const int a = (int)(e / (2 * chi_r));
  const R w = lam ? R(lam[a] * lam[a]) : R(1);
  M[(size_t)list[z] * per + e] = cscale(B[e], w);
}

}  // namespace mpsv

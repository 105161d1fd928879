// Gate-application kernels of the MPS simulator (arXiv:2303.03681, Methods,
// "MPS algorithm for quantum circuit simulation").
//
// Bond dimensions live in device memory (chi[b], b = 0..n); every kernel
// reads the dimensions it needs, so a whole gate sequence is issued without a
// host round trip and can be captured in a CUDA graph.  Grids are sized for
// the bond capacities; blocks past the actual dimensions return at once.
//
// A two-qubit gate on sites (q, q+1) runs two kernels (three where the tensor
// cores or, after an FP32 SVD, g3_kernel compute B~_q):
//   theta_kernel  C[(a_l,i),(j,a_r)] = sum Q[ij,i'j'] B_q[a_l,i',a_m] B_{q+1}[a_m,j',a_r];
//   svd_kernel    (svd_jacobi.cuh) SVD of lam_q[a_l] C (Eq. tildeC), truncation,
//                 B~_{q+1} = V (first k rows), lam_{q+1} = s[:k] / ||s[:k]||,
//                 B~_q = C V^dagger / ||s[:k]|| (Eq. Bl with the unscaled C).
#pragma once

#include "common.cuh"
#include "dfloat.cuh"

namespace mpsv {

constexpr int kTile = 16;

// Tile elements and accumulators of the CUDA-core complex contractions
// (theta, G3, the environments).  Complex64 states multiply-add in FP32.
// Complex128 states hold their shared-memory tiles as double-float values
// (converted once per tile load) and accumulate with exact heads plus FP32
// error terms (CAcc, packed) on the FP32 pipes: this part executes FP64 at 2 FMA
// per clock per SM against 128 FP32, and a double-float multiply-add costs
// 13 FP32 operations per real product (relative error about K 2^-47 of the
// sum of |terms| for K products, 1e-12 at K = 128).
template <typename R> struct Mac;
template <> struct Mac<float> {
  using Elem = float2;
  struct Acc {
    float2 v = make_float2(0.f, 0.f);
  };
  static __device__ __forceinline__ Elem load(float2 x) { return x; }
  static __device__ __forceinline__ Elem zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ void fma(Acc& a, Elem x, Elem y) { cfma(a.v, x, y); }    // += x y
  static __device__ __forceinline__ void fmac(Acc& a, Elem x, Elem y) { cfmac(a.v, x, y); }  // += conj(x) y
  static __device__ __forceinline__ float2 value(const Acc& a) { return a.v; }       // of fma sums
  static __device__ __forceinline__ float2 value_conj(const Acc& a) { return a.v; }  // of fmac sums
};
template <> struct Mac<double> {
  using Elem = Cff;
  using Acc = CAcc;
  static __device__ __forceinline__ Elem load(double2 x) { return cff_split(x); }
  static __device__ __forceinline__ Elem zero() { return Cff{mk2(0.f, 0.f), mk2(0.f, 0.f)}; }
  static __device__ __forceinline__ void fma(Acc& a, Elem x, Elem y) { a.add(x, y); }
  static __device__ __forceinline__ void fmac(Acc& a, Elem x, Elem y) { a.add(x, y); }
  static __device__ __forceinline__ double2 value(const Acc& a) { return a.value(); }
  static __device__ __forceinline__ double2 value_conj(const Acc& a) { return a.value_conj(); }
};

// ---------------------------------------------------------------------------
// reset to a computational basis state (chi = 1 everywhere)
// ---------------------------------------------------------------------------
template <typename R>
__global__ void reset_kernel(cplx<R>* __restrict__ B, const size_t* __restrict__ site_off,
                             double* __restrict__ lam, const size_t* __restrict__ lam_off,
                             int* __restrict__ chi, const uint8_t* __restrict__ bits, int n,
                             DevReport* __restrict__ rep) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) {
    cplx<R>* b = B + site_off[t];
    int bit = bits ? (bits[t] & 1) : 0;
    b[0] = cmk<R>(bit ? R(0) : R(1), R(0));
    b[1] = cmk<R>(bit ? R(1) : R(0), R(0));
  }
  if (t <= n) {
    chi[t] = 1;
    lam[lam_off[t]] = 1.0;
  }
  if (t == 0) {
    rep->discarded_weight = 0.0;
    rep->min_kept_sv = 1.0;
    rep->inv_norm = 1.0;
    rep->max_chi = 1;
    rep->degenerate_cuts = 0;
    rep->not_converged = 0;
    rep->max_sweeps = 0;
    rep->two_qubit_gates = 0;
    rep->svd_flops = 0.0;
    rep->tc_error = 0;
    rep->sweeps_fp32 = rep->sweeps_fp64 = 0;
    for (int i = 0; i < 4; ++i) rep->phase_cycles[i] = 0.0;
  }
}

// ---------------------------------------------------------------------------
// theta = B_q B_{q+1}; gate (G1 + G2; the SVD applies the lam scaling as it loads)
// ---------------------------------------------------------------------------
// The gate's entries for theta_tile, by the block's first 16 threads (one load
// each that hides behind the first tile's; read where they are used they added
// a load's latency to every gate).  The tile loop's barrier stands between.
template <typename R> struct GateTile {
  cplx<R> u[16];
  bool real;  // every imaginary part is zero
};
template <typename R>
__device__ __forceinline__ void load_gate(const DevGate* gate, int tid, GateTile<R>& g) {
  if (tid >= 32) return;
  const double2 z = tid < 16 ? __ldcg(gate->u + tid) : make_double2(0.0, 0.0);
  if (tid < 16) g.u[tid] = ccast<cplx<R>>(z);
  const bool im = __any_sync(0xffffffffu, (__double_as_longlong(z.y) << 1) != 0);
  if (tid == 0) g.real = !im;
}

// One 16 x 16 tile (a_l, a_r) with both physical indices, by 256 threads (tx,
// ty).  g: the gate in shared memory.  sL, sR: the group's tiles, 2 x 16 x 17 entries each.  Every thread of
// the block calls it (act false: no tile, only the barriers).  The site tensors
// are read past L1: a run of gates changes them between calls.
template <typename R>
__device__ __forceinline__ void theta_tile(const cplx<R>* __restrict__ Bl, const cplx<R>* __restrict__ Br,
                                           const GateTile<R>& g, int chi_l, int chi_m, int chi_r, int al0,
                                           int ar0, int tx, int ty, bool act, typename Mac<R>::Elem (*sL)[kTile][kTile + 1],
                                           typename Mac<R>::Elem (*sR)[kTile][kTile + 1], cplx<R>* __restrict__ Cm) {
  using C = cplx<R>;
  using MT = Mac<R>;
  using E = typename MT::Elem;
  typename MT::Acc acc[2][2];
  const int al = al0 + ty, ar = ar0 + tx;
  act = act && al0 < chi_l && ar0 < chi_r;
  const bool mine = act && al < chi_l && ar < chi_r;
  // the next tiles are loaded while these are summed: a small theta is a chain
  // of its chi_m / 16 load latencies (28-qubit UCCSD 53.8 -> 53.0 ms)
  C l0 = cmk<R>(0, 0), l1 = l0, r0 = l0, r1 = l0;
  auto fetch = [&](int m0) {
    const int mm = m0 + tx, mr = m0 + ty;
    const bool ok = al < chi_l && mm < chi_m, okr = mr < chi_m && ar < chi_r;
    l0 = ok ? __ldcg(Bl + (size_t)(al * 2 + 0) * chi_m + mm) : cmk<R>(0, 0);
    l1 = ok ? __ldcg(Bl + (size_t)(al * 2 + 1) * chi_m + mm) : cmk<R>(0, 0);
    r0 = okr ? __ldcg(Br + (size_t)(mr * 2 + 0) * chi_r + ar) : cmk<R>(0, 0);
    r1 = okr ? __ldcg(Br + (size_t)(mr * 2 + 1) * chi_r + ar) : cmk<R>(0, 0);
  };
  if (act) fetch(0);
  for (int m0 = 0; m0 < chi_m; m0 += kTile) {
    if (act) {
      sL[0][ty][tx] = MT::load(l0);
      sL[1][ty][tx] = MT::load(l1);
      sR[0][ty][tx] = MT::load(r0);
      sR[1][ty][tx] = MT::load(r1);
    }
    __syncthreads();
    if (act && m0 + kTile < chi_m) fetch(m0 + kTile);
    if (mine) {
      const int kend = min(kTile, chi_m - m0);
#pragma unroll 4
      for (int kk = 0; kk < kend; ++kk) {
        const E x0 = sL[0][ty][kk], x1 = sL[1][ty][kk];
        const E y0 = sR[0][kk][tx], y1 = sR[1][kk][tx];
        MT::fma(acc[0][0], x0, y0);
        MT::fma(acc[0][1], x0, y1);
        MT::fma(acc[1][0], x1, y0);
        MT::fma(acc[1][1], x1, y1);
      }
    }
    __syncthreads();
  }
  if (!mine) return;
  // the gate on (i', j'), in the storage precision.  Complex128 takes FP64
  // multiply-adds, two per clock and SM: the 64 of a thread are as long as a
  // 16-column theta's sums, so a real gate (nine in ten of a UCCSD circuit) takes
  // its 32 only (28-qubit UCCSD 54.2 -> 52.5 ms; in double-float, which would
  // round theta to 2^-47 once more, 52.3)
  const int n = 2 * chi_r;
  C th[2][2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) th[i][j] = MT::value(acc[i][j]);
  auto apply = [&](auto term) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        C out = cmk<R>(0, 0);
#pragma unroll
        for (int ip = 0; ip < 2; ++ip)
#pragma unroll
          for (int jp = 0; jp < 2; ++jp) term(out, g.u[(2 * i + j) * 4 + 2 * ip + jp], th[ip][jp]);
        Cm[(size_t)(2 * al + i) * n + j * chi_r + ar] = out;
      }
    }
  };
  if (sizeof(R) == 8 && g.real)
    apply([](C& out, C u, C t) {
      out.x = fma(u.x, t.x, out.x);
      out.y = fma(u.x, t.y, out.y);
    });
  else
    apply([](C& out, C u, C t) { cfma(out, u, t); });
}

template <typename R>
__global__ void __launch_bounds__(kTile* kTile)
    theta_kernel(const cplx<R>* __restrict__ Bl, const cplx<R>* __restrict__ Br,
                 const DevGate* __restrict__ gate, const int* __restrict__ chi, int q, cplx<R>* __restrict__ Cm) {
  __shared__ typename Mac<R>::Elem sL[2][kTile][kTile + 1];
  __shared__ typename Mac<R>::Elem sR[2][kTile][kTile + 1];
  // launched while the gate before may still run (gate by gate on a stream):
  // its results are read after this, and past L1
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  const int chi_l = __ldcg(chi + q), chi_r = __ldcg(chi + q + 2);
  const int al0 = blockIdx.y * kTile, ar0 = blockIdx.x * kTile;
  if (al0 >= chi_l || ar0 >= chi_r) return;
  __shared__ GateTile<R> s_g;
  load_gate<R>(gate, threadIdx.y * kTile + threadIdx.x, s_g);
  theta_tile<R>(Bl, Br, s_g, chi_l, __ldcg(chi + q + 1), chi_r, al0, ar0, threadIdx.x, threadIdx.y, true, sL, sR, Cm);
}

// ---------------------------------------------------------------------------
// B~_q = C B~_{q+1}^dagger / ||s[:k]||  (G3, Eq. Bl)
// ---------------------------------------------------------------------------
template <typename R>
__global__ void __launch_bounds__(kTile* kTile)
    g3_kernel(const cplx<R>* __restrict__ Cm, const cplx<R>* __restrict__ Bn, const int* __restrict__ chi, int q,
              const DevReport* __restrict__ rep, cplx<R>* __restrict__ Bout) {
  using C = cplx<R>;
  using MT = Mac<R>;
  using E = typename MT::Elem;
  const int chi_l = chi[q], k = chi[q + 1], chi_r = chi[q + 2];
  const int m = 2 * chi_l, n = 2 * chi_r;
  const int r0 = blockIdx.y * kTile, a0 = blockIdx.x * kTile;
  if (r0 >= m || a0 >= k) return;
  const int tx = threadIdx.x, ty = threadIdx.y;
  __shared__ E sA[kTile][kTile + 1];
  __shared__ E sB[kTile][kTile + 1];  // conj(B~_{q+1})
  typename MT::Acc acc;
  for (int c0 = 0; c0 < n; c0 += kTile) {
    const int c = c0 + tx;
    sA[ty][tx] = (r0 + ty < m && c < n) ? MT::load(Cm[(size_t)(r0 + ty) * n + c]) : MT::zero();
    sB[ty][tx] = (a0 + ty < k && c < n) ? MT::load(cconj(Bn[(size_t)(a0 + ty) * n + c])) : MT::zero();
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < kTile; ++kk) MT::fma(acc, sA[ty][kk], sB[tx][kk]);
    __syncthreads();
  }
  const int r = r0 + ty, a = a0 + tx;
  if (r < m && a < k) {
    const R inv = R(rep->inv_norm);
    const C v = MT::value(acc);
    Bout[(size_t)r * k + a] = cmk<R>(v.x * inv, v.y * inv);
  }
}

// ---------------------------------------------------------------------------
// one-qubit gate (exact, keeps the canonical form)
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ void gate1_entry(cplx<R>* __restrict__ B, const DevGate* __restrict__ gate, int chi_r,
                                            int t) {
  using C = cplx<R>;
  const int al = t / chi_r, ar = t % chi_r;
  C* p0 = B + (size_t)(al * 2 + 0) * chi_r + ar;
  C* p1 = B + (size_t)(al * 2 + 1) * chi_r + ar;
  const C b0 = __ldcg(p0), b1 = __ldcg(p1);
  C n0 = cmk<R>(0, 0), n1 = cmk<R>(0, 0);
  cfma(n0, ccast<C>(gate->u[0]), b0);
  cfma(n0, ccast<C>(gate->u[1]), b1);
  cfma(n1, ccast<C>(gate->u[2]), b0);
  cfma(n1, ccast<C>(gate->u[3]), b1);
  *p0 = n0;
  *p1 = n1;
}

template <typename R>
__global__ void gate1_kernel(cplx<R>* __restrict__ B, const DevGate* __restrict__ gate, const int* __restrict__ chi,
                             int q) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < chi[q] * chi[q + 1]) gate1_entry<R>(B, gate, chi[q + 1], t);
}

// ---------------------------------------------------------------------------
// bind template angles: u = exp(i phi) M+ + exp(-i phi) M-
// ---------------------------------------------------------------------------
static __global__ void bind_kernel(const DevTmplGate* __restrict__ tmpl, int n_gates, const double* __restrict__ theta,
                                   DevGate* __restrict__ out) {
  const int g = blockIdx.x;
  if (g >= n_gates) return;
  const DevTmplGate& t = tmpl[g];
  const double phi = t.param >= 0 ? t.coeff * theta[t.param] : 0.0;
  double s, c;
  sincos(phi, &s, &c);
  const int e = threadIdx.x;
  if (e < 16) {
    const double2 a = t.mp[e], b = t.mm[e];
    // (c + i s) a + (c - i s) b
    double2 u;
    u.x = c * (a.x + b.x) - s * (a.y - b.y);
    u.y = c * (a.y + b.y) + s * (a.x - b.x);
    out[g].u[e] = u;
  }
  if (e == 0) {
    out[g].q = t.q;
    out[g].arity = t.arity;
  }
}

}  // namespace mpsv

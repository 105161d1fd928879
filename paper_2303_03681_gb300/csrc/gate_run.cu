// Runs of gates in one launch: the theta contraction, the truncation SVD and
// B~_q of every two-qubit gate, and the one-qubit gates, one after another on
// one CTA or one thread-block cluster.
//
// A UCCSD circuit is a chain of gates on small bonds (the median theta of the
// 50-qubit workload is 16 x 16), each of which waits for the one before it.
// Launched one by one, many evaluations at once are bound by the hardware
// queues that their streams share and by the rate at which the host threads
// can launch.  Here the bond dimensions and the report stay on the SM and a
// whole circuit is at most three launches: 32 evaluations of a 16-qubit UCCSD
// circuit take 103 ms instead of 227 with the default 8 hardware queues, 104
// instead of 121 with 32 (gate_by_gate_streams in energy.cu has the rule and the
// other figures).  What bounds a run is the chain of dependent steps inside
// its SVDs.
//
// Tiers.  A theta gets 1, 4 or 8 CTAs by its sizes alone (svd_team_size), so
// its arithmetic does not depend on the launch.  The runs are issued one
// after another: a launch of one CTA goes on until a gate needs more, then one of 4
// CTAs, then one of 8 where the capacities ask for it; each starts where the
// one before it stopped (progress) and returns at once when nothing is
// left.  A launch of one CTA holds one SM, so that many evaluations of
// small fragments run side by side.
#include <algorithm>
#include <mutex>

#include "gate_kernels.cuh"
#include "internal.h"
#include "svd_launch.cuh"

namespace mpsv {

namespace {

// 12 warps: 168 registers a thread, at which the one-CTA bodies spill 32 to 40
// bytes a thread and the cluster's double-float one 350 (1,100 read).  One
// evaluation takes 84.8 ms, with 8 warps 86.3 and with 16 (128 registers) 88.9.
constexpr int kRunThreads = 384;

struct RunArgs {
  const DevGate* gates;
  int n_gates;
  int svd_fp64;
  void* B;
  const size_t* site_off;
  double* lam;
  const size_t* lam_off;
  const int* cap;  // bond capacities
  int* chi;
  DevReport* rep;
  void* C;
  char* ws;
  int* progress;  // gates done
  int first;      // start at gate 0
  SvdParams p;
};

// CTAs that a gate does not need keep the cluster barriers in step: they
// count them until the number that CTA 0 has told them for this gate.  (A
// plain flag could be seen one barrier early.)
__device__ __forceinline__ void follow(volatile long long* done, int g) {
  for (int n = 1;; ++n) {
    cg::this_cluster().sync();
    const long long d = *done;
    if ((int)(d >> 32) == g && (int)d == n) return;
  }
}

template <typename R>
__device__ __forceinline__ void run_theta(const RunArgs& a, const DevGate* g, int q, int me, int P) {
  using E = typename Mac<R>::Elem;
  using Tile = E(*)[kTile][kTile + 1];
  const cplx<R>* B = static_cast<const cplx<R>*>(a.B);
  const int chi_l = __ldcg(a.chi + q), chi_m = __ldcg(a.chi + q + 1), chi_r = __ldcg(a.chi + q + 2);
  __shared__ GateTile<R> s_g;
  load_gate<R>(g, threadIdx.x, s_g);
  // 256 of the threads take the tiles; the others join the barriers only
  const int t = threadIdx.x & 255;
  E* base = reinterpret_cast<E*>(svd_smem);
  const int tr = (chi_r + kTile - 1) / kTile, tiles = tr * ((chi_l + kTile - 1) / kTile);
  for (int tile = me; tile < tiles; tile += P)
    theta_tile<R>(B + a.site_off[q], B + a.site_off[q + 1], s_g, chi_l, chi_m, chi_r, (tile / tr) * kTile,
                  (tile % tr) * kTile, t & 15, t >> 4, threadIdx.x < 256, reinterpret_cast<Tile>(base),
                  reinterpret_cast<Tile>(base + 2 * kTile * (kTile + 1)), static_cast<cplx<R>*>(a.C));
}

// Not inlined: each instance gets its own registers.
template <class A, class R, class Team>
__device__ __noinline__ void run_two_qubit(const RunArgs& a, Team& tm, const DevGate* g, int q, int* s_chi,
                                              DevReport* rep) {
  run_theta<R>(a, g, q, tm.me, tm.P);
  tm.barrier();
  cplx<R>* B = static_cast<cplx<R>*>(a.B);
  svd_body<A, R, Team, false>(tm, static_cast<const cplx<R>*>(a.C), a.lam + a.lam_off[q], 2 * __ldcg(a.chi + q),
                              2 * __ldcg(a.chi + q + 2), a.p, B + a.site_off[q + 1], a.lam + a.lam_off[q + 1], s_chi, rep,
                              B + a.site_off[q], a.ws);
}

// kCluster: launches of several CTAs.
template <typename R, bool kCluster>
__global__ void __launch_bounds__(kRunThreads, 1) gate_run_kernel(RunArgs a) {
  __shared__ float2 s_mail[2 * 16];
  __shared__ DevReport s_rep;
  __shared__ long long s_done;
  __shared__ int s_chi;
  const int Pl = kCluster ? (int)cg::this_cluster().num_blocks() : 1;
  const int me = kCluster ? (int)cg::this_cluster().block_rank() : 0;
  const int tid = threadIdx.x, T = blockDim.x;
  if (tid == 0) {
    s_done = -1;
    if (me == 0) s_rep = *a.rep;
  }
  int g = a.first ? 0 : __ldcg(a.progress);
  if (kCluster)
    cg::this_cluster().sync();  // every CTA has read the progress and runs
  else
    __syncthreads();
  for (; g < a.n_gates; ++g) {
    const DevGate* gate = a.gates + g;
    const int q = gate->q;
    if (gate->arity == 1) {
      // exact, keeps the canonical form
      if (me == 0) {
        using C = cplx<R>;
        C* B = static_cast<C*>(a.B) + a.site_off[q];
        const int chi_l = __ldcg(a.chi + q), chi_r = __ldcg(a.chi + q + 1);
        for (int t = tid; t < chi_l * chi_r; t += T) gate1_entry<R>(B, gate, chi_r, t);
      }
    } else {
      const int m = 2 * __ldcg(a.chi + q), n = 2 * __ldcg(a.chi + q + 2);
      const bool f64 = a.svd_fp64 == 2 || 2 * a.cap[q + 2] < 32;
      const int P = f64 ? svd_team_size<ArF64>(m, n, Pl) : svd_team_size<ArDF>(m, n, Pl);
      if (P == 0) break;  // for a launch of more CTAs
      if (me < P) {
        int barriers = 0;
        if (P == 1) {
          OneTeam tm;
          if (f64)
            run_two_qubit<ArF64, R>(a, tm, gate, q, &s_chi, &s_rep);
          else
            run_two_qubit<ArDF, R>(a, tm, gate, q, &s_chi, &s_rep);
        } else if constexpr (kCluster) {
          ClusterTeam tm{me, P, s_mail};
          if (f64)
            run_two_qubit<ArF64, R>(a, tm, gate, q, &s_chi, &s_rep);
          else
            run_two_qubit<ArDF, R>(a, tm, gate, q, &s_chi, &s_rep);
          barriers = tm.barriers;
        }
        __syncthreads();
        if (me == 0 && tid == 0) a.chi[q + 1] = s_chi;
        if (kCluster && me == 0 && P > 1 && tid >= P && tid < Pl)
          *cg::this_cluster().map_shared_rank(&s_done, tid) = ((long long)g << 32) | (barriers + 1);
      } else if (kCluster && P > 1) {
        follow(&s_done, g);
        continue;
      }
    }
    // the gate's results before the next gate's reads
    if (kCluster)
      cg::this_cluster().sync();
    else
      __syncthreads();
  }
  if (me == 0 && tid == 0) {
    *a.rep = s_rep;
    *a.progress = g;
  }
}

template <typename R> cudaError_t run_attrs() {
  static std::mutex mu;
  static uint64_t done = 0;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> g(mu);
  const uint64_t bit = 1ull << (dev & 63);
  if (done & bit) return cudaSuccess;
  cudaError_t e =
      cudaFuncSetAttribute(gate_run_kernel<R, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSvdSmemLimit);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gate_run_kernel<R, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSvdSmemLimit);
  if (e == cudaSuccess) done |= bit;
  return e;
}

template <typename R> void launch_run(mps_state* st, const DevGate* d_gates, size_t n, int P) {
  (void)run_attrs<R>();
  RunArgs a;
  a.gates = d_gates;
  a.n_gates = (int)n;
  a.svd_fp64 = st->cfg.svd_fp64;
  a.B = st->d_B;
  a.site_off = st->d_site_off;
  a.lam = st->d_lam;
  a.lam_off = st->d_lam_off;
  a.cap = st->d_cap;
  a.chi = st->d_chi;
  a.rep = st->d_rep;
  a.C = st->d_C;
  a.ws = st->d_svd;
  a.progress = st->d_cap + st->n + 1;
  a.p = svd_params(st);
  a.first = P == 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(P);
  cfg.blockDim = dim3(kRunThreads);
  cfg.dynamicSmemBytes = P == 1 ? st->run_smem : kSvdSmemLimit;
  cfg.stream = st->ctx->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = P;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (P == 1)
    cudaLaunchKernelEx(&cfg, gate_run_kernel<R, false>, a);
  else
    cudaLaunchKernelEx(&cfg, gate_run_kernel<R, true>, a);
}

// CTAs of a bond's largest theta (0: a grid) and the single CTA's shared memory.
template <class A> void bond_plan(int m, int n, int& P, size_t& smem) {
  P = svd_team_size<A>(m, n, 8);
  smem = n <= kSvdSingleCols ? SvdSmem<A>::bytes_one(m, n) : kSvdSmemLimit;
}

}  // namespace

void run_prime() {
  (void)run_attrs<float>();
  (void)run_attrs<double>();
}

void run_setup(mps_state* st) {
  size_t smem = (size_t)4 * kTile * (kTile + 1) * sizeof(Cff);  // theta's tiles
  st->run_p.assign(st->n, 0);
  for (int q = 0; q + 1 < st->n; ++q) {
    const int m = 2 * st->cap[q], n = 2 * st->cap[q + 2];
    size_t need = 0;
    if (svd_arith(st->cfg.svd_fp64, n) == SVD_F64)
      bond_plan<ArF64>(m, n, st->run_p[q], need);
    else
      bond_plan<ArDF>(m, n, st->run_p[q], need);
    smem = std::max(smem, need);
  }
  st->run_smem = smem;
}

bool run_tier(mps_state* st, const DevGate* d_gates, size_t n, int p_max, int tier) {
  const int P = tier == 0 ? 1 : 2 << tier;  // 1, 4, 8
  if (P > p_max) return false;
  if (st->fp32)
    launch_run<float>(st, d_gates, n, P);
  else
    launch_run<double>(st, d_gates, n, P);
  return true;
}

}  // namespace mpsv

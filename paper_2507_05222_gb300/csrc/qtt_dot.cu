// Overlap <a, b> of two trains in one launch (norms, energies and overlaps of a run).
//
// The train is contracted from both ends at once: E_L(a, b) over sites 0, 1, ... and E_R(a, b) over
// sites n - 1, n - 2, ..., joined by one sum over the middle bond.  A step takes one site on
// each side, in two phases,
//   left   T(b, s, a') = sum_a  E_L(a, b) A(a, s, a')     E_L'(a', b') = sum_{b, s} T(b, s, a') B(b, s, b')
//   right  T(a, s, b') = sum_a' A(a, s, a') E_R(a', b')   E_R'(a, b)   = sum_{s, b'} T(a, s, b') B(b, s, b')
// with a barrier after each; several lanes share an output where outputs are few.  What bounds it is
// the chain of n phases (L2 latency, an FP64 shuffle sum, the barrier), not the arithmetic: below
// the line in dot_fused a 16-CTA cluster runs it (hardware barrier, about 0.2 us), above it one
// cooperative grid (1.3 us a barrier, but all SMs' FP64 units).  Contracting site by site took two
// launches a site; both are timed at dot_fused.
#include <cooperative_groups.h>

#include <algorithm>

#include "qtt_algebra.h"

namespace cgrp = cooperative_groups;

namespace qtt {

namespace {

constexpr int DT_THREADS = 256;
constexpr int DT_MAX_N = 64;
constexpr int DT_CLUSTER = 16;
constexpr int DT_CLUSTER_BOND = 32;     // largest bond of the cluster variant
constexpr int DT_MAX_BOND = 64;

struct DotArgs {
  int n, d;
  int ab[DT_MAX_N + 1], bb[DT_MAX_N + 1];
  int64_t ao[DT_MAX_N], bo[DT_MAX_N];
  const double* A;
  const double* B;
  double* ws;           // per side: E, E', T
  int64_t es, ts;       // sizes of E and T
  double* out;          // the value; 0, or 1 where the grid variant gave up waiting
  unsigned int* bar;    // grid variant: arrivals, whether a CTA gave up
  unsigned long long limit_ns;
};

__device__ __forceinline__ unsigned long long dt_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid barrier, bounded by the context's wait limit; false once a CTA gave up.
__device__ bool dt_grid_sync(const DotArgs& a, unsigned int& target, int* flag) {
  target += gridDim.x;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(a.bar), "r"(1u) : "memory");
    const unsigned long long t0 = dt_ns();
    const unsigned int mask = a.limit_ns < 100000ull ? 0u : 255u;
    unsigned int spins = 0, v;
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.bar) : "memory");
      if (v >= target) break;
      if ((++spins & mask) == 0u) {
        if (*reinterpret_cast<const volatile unsigned int*>(a.bar + 1)) break;
        if (dt_ns() - t0 > a.limit_ns) {
          atomicExch(a.bar + 1, 1u);
          break;
        }
      }
    }
    __threadfence();
    *flag = int(*reinterpret_cast<const volatile unsigned int*>(a.bar + 1));
  }
  __syncthreads();
  return *flag == 0;
}

// out(o) = sum_k X(xo(o) + k-offset) Y(...) for o = 0 .. no-1 handled by this side's threads: t0 of nt
// threads, LPO lanes an output.  k = (k1, k2), k2 < n2 fastest; x and y advance by (x1, x2), (y1, y2).
// The output o = (o1, o2, o3) with o3 fastest (dims m2, m3): strides ox*, oy*.
struct DotPhase {
  const double* x;
  const double* y;
  double* out;
  bool xl2, yl2;              // operand written in this launch: read through L2
  int no, m2, m3, n1, n2;
  int x1, x2, y1, y2, ox1, ox2, ox3, oy1, oy2, oy3;
};

template <int LPO>
__device__ void dt_phase_lpo(const DotPhase& p, int t, int nt) {
  const int lane = t % LPO;
  const int K = p.n1 * p.n2;
  const int rounds = (p.no * LPO + nt - 1) / nt;     // every lane of a warp takes every round
  for (int r = 0; r < rounds; ++r) {
    const int o = (t + r * nt) / LPO;
    double s0 = 0.0, s1 = 0.0;
    if (o < p.no) {
      const int o3 = o % p.m3, o2 = (o / p.m3) % p.m2, o1 = o / (p.m3 * p.m2);
      const double* x = p.x + o1 * p.ox1 + o2 * p.ox2 + o3 * p.ox3;
      const double* y = p.y + o1 * p.oy1 + o2 * p.oy2 + o3 * p.oy3;
#pragma unroll 4
      for (int k = lane; k < K; k += LPO) {
        const int k1 = k / p.n2, k2 = k - k1 * p.n2;
        const double* xp = x + k1 * p.x1 + k2 * p.x2;
        const double* yp = y + k1 * p.y1 + k2 * p.y2;
        const double xv = p.xl2 ? __ldcg(xp) : __ldg(xp), yv = p.yl2 ? __ldcg(yp) : __ldg(yp);
        const double s = s0;
        s0 = s1;
        s1 = fma(xv, yv, s);                          // two partial sums in turn
      }
    }
    double s = s0 + s1;
    for (int off = LPO / 2; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (o < p.no && lane == 0) p.out[o] = s;
  }
}

__device__ void dt_phase(const DotPhase& p, int t, int nt) {
  const int K = p.n1 * p.n2;
  int lpo = 1;
  while (lpo < 32 && p.no * lpo * 2 <= nt && lpo * 2 <= K) lpo *= 2;
  switch (lpo) {
    case 1: dt_phase_lpo<1>(p, t, nt); break;
    case 2: dt_phase_lpo<2>(p, t, nt); break;
    case 4: dt_phase_lpo<4>(p, t, nt); break;
    case 8: dt_phase_lpo<8>(p, t, nt); break;
    case 16: dt_phase_lpo<16>(p, t, nt); break;
    default: dt_phase_lpo<32>(p, t, nt); break;
  }
}

template <bool CLUSTER>
__global__ void __launch_bounds__(DT_THREADS) k_dot_fused(const __grid_constant__ DotArgs a) {
  __shared__ int flag;
  __shared__ double red[DT_THREADS / 32];
  unsigned int target = 0;
  auto barrier = [&]() {
    if (CLUSTER) {
      __threadfence();
      cgrp::this_cluster().sync();
      return true;
    }
    return dt_grid_sync(a, target, &flag);
  };
  const int G = gridDim.x, half = G / 2, tid = threadIdx.x;
  const bool right = int(blockIdx.x) >= half;
  const int nb = right ? G - half : half;
  const int t = (right ? int(blockIdx.x) - half : int(blockIdx.x)) * DT_THREADS + tid, nt = nb * DT_THREADS;
  double* E = a.ws + (right ? 2 * a.es + a.ts : 0);
  double* En = E + a.es;
  double* T = En + a.es;
  const int d = a.d, nl = a.n / 2, nr = a.n - nl;      // sites of the left and of the right half
  if (t == 0) E[0] = 1.0;
  bool ok = barrier();
  for (int step = 0; step < nr && ok; ++step) {
    const bool live = right || step < nl;
    const int k = right ? a.n - 1 - step : step;
    const int a0 = a.ab[k], a1 = a.ab[k + 1], b0 = a.bb[k], b1 = a.bb[k + 1];
    const double* Ak = a.A + a.ao[k];
    const double* Bk = a.B + a.bo[k];
    if (live) {
      DotPhase p;
      p.out = T;
      if (!right) {          // T(b, s, a') = sum_a E(a, b) A(a, s, a')
        p.x = E; p.xl2 = true; p.y = Ak; p.yl2 = false;
        p.no = b0 * d * a1; p.m2 = d; p.m3 = a1; p.n1 = 1; p.n2 = a0;
        p.x1 = 0; p.x2 = b0; p.y1 = 0; p.y2 = d * a1;
        p.ox1 = 1; p.ox2 = 0; p.ox3 = 0; p.oy1 = 0; p.oy2 = a1; p.oy3 = 1;
      } else {               // T(a, s, b') = sum_a' A(a, s, a') E(a', b')
        p.x = Ak; p.xl2 = false; p.y = E; p.yl2 = true;
        p.no = a0 * d * b1; p.m2 = d; p.m3 = b1; p.n1 = 1; p.n2 = a1;
        p.x1 = 0; p.x2 = 1; p.y1 = 0; p.y2 = b1;
        p.ox1 = d * a1; p.ox2 = a1; p.ox3 = 0; p.oy1 = 0; p.oy2 = 0; p.oy3 = 1;
      }
      dt_phase(p, t, nt);
    }
    if (!(ok = barrier())) break;
    if (live) {
      DotPhase p;
      p.out = En;
      p.x = T; p.xl2 = true; p.y = Bk; p.yl2 = false; p.m2 = 1;
      if (!right) {          // E'(a', b') = sum_{b, s} T(b, s, a') B(b, s, b')
        p.no = a1 * b1; p.m3 = b1; p.n1 = 1; p.n2 = b0 * d;
        p.x1 = 0; p.x2 = a1; p.y1 = 0; p.y2 = b1;
        p.ox1 = 1; p.ox2 = 0; p.ox3 = 0; p.oy1 = 0; p.oy2 = 0; p.oy3 = 1;
      } else {               // E'(a, b) = sum_{s, b'} T(a, s, b') B(b, s, b')
        p.no = a0 * b0; p.m3 = b0; p.n1 = 1; p.n2 = d * b1;
        p.x1 = 0; p.x2 = 1; p.y1 = 0; p.y2 = 1;
        p.ox1 = d * b1; p.ox2 = 0; p.ox3 = 0; p.oy1 = 0; p.oy2 = 0; p.oy3 = d * b1;
      }
      dt_phase(p, t, nt);
      double* q = E;
      E = En;
      En = q;
    }
    if (!(ok = barrier())) break;
  }
  if (blockIdx.x != 0) return;
  // the left half made nl swaps, the right half nr
  const double* L = a.ws + (nl & 1 ? a.es : 0);
  const double* R = a.ws + 2 * a.es + a.ts + (nr & 1 ? a.es : 0);
  const int m = a.ab[nl] * a.bb[nl];
  double s = 0.0;
  for (int e = tid; e < m; e += DT_THREADS) s = fma(__ldcg(L + e), __ldcg(R + e), s);
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if ((tid & 31) == 0) red[tid >> 5] = s;
  __syncthreads();
  if (tid == 0) {
    double v = 0.0;
    for (int w = 0; w < DT_THREADS / 32; ++w) v += red[w];
    a.out[0] = v;
    a.out[1] = ok ? 0.0 : 1.0;
  }
}

// Whether the cluster variant is available.
bool dot_cluster_available() {
  bool ok = false;
  if (cudaFuncSetAttribute(k_dot_fused<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(DT_CLUSTER);
    cfg.blockDim = dim3(DT_THREADS);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = DT_CLUSTER;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int nclusters = 0;
    ok = cudaOccupancyMaxActiveClusters(&nclusters, k_dot_fused<true>, &cfg) == cudaSuccess && nclusters >= 1;
  }
  cudaGetLastError();
  return ok;
}

}  // namespace

// At most 64 sites and bonds up to 64: the cluster up to bond 32, the grid above (a call of mps_dot,
// us: 12 sites 130 -> 41 at bond 16, 145 -> 65 at bond 64; 20 sites 214 -> 64 at bond 16, 237 -> 89
// at bond 32 on the cluster, 278 -> 117 at bond 64 on the grid).  Above bond 64 the site-by-site
// path stays (its products reach the batched GEMM).
bool dot_fused(Ctx& c, const qtt_mps* x, const qtt_mps* y, double* out_dev) {
  const int n = x->n, d = x->d;
  if (n > DT_MAX_N) return false;
  int bond = 1;
  int64_t es = 1, ts = 1;
  for (int k = 0; k <= n; ++k) bond = std::max(bond, std::max(x->bonds[k], y->bonds[k]));
  if (bond > DT_MAX_BOND) return false;
  for (int k = 0; k <= n; ++k) es = std::max<int64_t>(es, int64_t(x->bonds[k]) * y->bonds[k]);
  for (int k = 0; k < n; ++k)
    ts = std::max<int64_t>(ts, d * std::max<int64_t>(int64_t(y->bonds[k]) * x->bonds[k + 1], int64_t(x->bonds[k]) * y->bonds[k + 1]));
  static const bool available = dot_cluster_available();   // once: the others of several threads wait for it
  const bool cluster = bond <= DT_CLUSTER_BOND && available;
  DotArgs a;
  a.n = n; a.d = d;
  for (int k = 0; k <= n; ++k) { a.ab[k] = x->bonds[k]; a.bb[k] = y->bonds[k]; }
  for (int k = 0; k < n; ++k) { a.ao[k] = x->off[k]; a.bo[k] = y->off[k]; }
  a.A = x->buf.p; a.B = y->buf.p;
  a.es = es; a.ts = ts;
  DBuf ws(&c, size_t(2 * (2 * es + ts))), bar(&c, 1);
  a.ws = ws.p;
  a.out = out_dev;
  a.bar = reinterpret_cast<unsigned int*>(bar.p);
  a.limit_ns = c.root->wait_ns;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(DT_THREADS);
  cfg.stream = c.stream;
  cudaLaunchAttribute at[1];
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (cluster) {
    cfg.gridDim = dim3(DT_CLUSTER);
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = DT_CLUSTER;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    QTT_CUDA(cudaLaunchKernelEx(&cfg, k_dot_fused<true>, a));
  } else {
    fill(c, bar.p, 1, 0.0);
    cfg.gridDim = dim3(unsigned(&c == c.root ? c.num_sms : std::max(2, c.num_sms / 2)));
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    QTT_CUDA(cudaLaunchKernelEx(&cfg, k_dot_fused<false>, a));
  }
  after_launch(c, "dot_fused");
  return true;
}

}  // namespace qtt

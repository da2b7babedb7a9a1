// Local CG solve of a small ALS site (Sec. II.A.4) in one thread-block cluster.
//
// A team of CS CTAs owns a row c (or several) of the unknown x[c, s, e] and applies the operator to it:
//   T1[w, t, b] = sum_a L[c, w, a] P[a, t, b],  T2[s, v, b] = sum_{w,t} T1[w, t, b] W[w, s, t, v]
//     for the CTA's own b, written into every team member's shared memory (DSMEM); barrier;
//   Ap[c, s, e] = sum_{v,b} T2[s, v, b] R[e, v, b] for the CTA's own e.
// The CTA that computes Ap[c, s, e] owns x, r, p, Ap and the preconditioner of those elements in
// its shared memory.  The recurrences are those of qtt_cg.cu with two barriers an iteration: the first
// carries the sums of p.Ap, the second those of r.r and r.z together with z, from which every CTA
// forms the next p = z + beta p of the b that it needs in its own shared memory.
//
// What bounds it: barriers and FP64 latency (64 clocks an operation, 110 a shuffle-sum level).
// qtt_cg.cu's kernels take three to four grid barriers of 1.3 us and five block reductions an
// iteration; a cluster of up to 16 CTAs has a hardware barrier of 0.2 us, which cannot be left waiting
// for a CTA that is not resident.  Timed at cg_team_plan.
#include <cooperative_groups.h>

#include <algorithm>
#include <map>
#include <mutex>

#include "qtt_algebra.h"

namespace cgrp = cooperative_groups;

namespace qtt {

namespace {

constexpr int TM_THREADS = 256;
constexpr int TM_SUMS = 3;        // at most: b.b, r.r, r.z
constexpr int TM_POISON = -(1 << 29);
constexpr size_t TM_SMEM = 200 * 1024;
constexpr int TM_CLUSTER = 16, TM_ELEMS = 256;

struct TeamArgs {
  int r0, r1, w0, w1, d, iters;
  int cs, teams, bw, ew, rows;    // team size, teams, b and e per CTA, rows c per team
  int rres;                       // R's rows resident in shared memory
  const double* tol;
  const double* L;
  const double* W;
  const double* R;
  const double* b;
  const double* xin;
  double* xout;
  double* z;                      // published D r (r0, d, r1)
  double* part;                   // 2 x TM_SUMS x gridDim.x: the sums of the two barriers
  unsigned long long limit_ns;
  int* total;
  double* flops;
  double fpi;
};

__device__ __forceinline__ unsigned long long tm_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// The hardware barrier needs no bound; a wait beyond the limit is reported in the first CTA's err
// all the same.
__device__ void tm_sync(const TeamArgs& a, int* err) {
  cgrp::cluster_group cl = cgrp::this_cluster();
  const unsigned long long t0 = threadIdx.x == 0 ? tm_ns() : 0ull;
  __threadfence();
  cl.sync();
  if (threadIdx.x == 0 && tm_ns() - t0 > a.limit_ns) *cl.map_shared_rank(err, 0) = 1;
}

__device__ __forceinline__ double tm_warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Lanes that share an output of the last contraction: as many as the threads allow, at most the 16 of
// qtt_cg.cu's stage B.
__device__ __forceinline__ int tm_lanes(int outs) {
  int l = 1;
  while (l < 16 && outs * l * 2 <= TM_THREADS) l *= 2;
  return l;
}

// sum_k x[k sx] y[k sy] over lanes l, l + nl, ..., then over the lanes.
template <bool YG>
__device__ __forceinline__ double tm_dot(const double* x, int sx, const double* y, int sy, int K, int l, int nl, bool in) {
  double s = 0.0;
  if (in)
    for (int k = l; k < K; k += nl) s = fma(x[k * sx], YG ? __ldg(y + k * sy) : y[k * sy], s);
  for (int o = nl >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

struct TeamSmem {
  double *P, *L, *W, *T1, *T2, *R, *x, *r, *p, *Ap, *di;
};

// P[a, t, b of this CTA] <- V[a, t, b] + beta P, V (r0, d, r1) in global memory, read through L2 (other
// CTAs write z in this launch).  beta = 0 takes V alone.
__device__ void tm_direction(const TeamArgs& a, const TeamSmem& s, const double* V, double beta, int rank) {
  const int bw = a.bw, b0 = rank * bw, nbw = max(0, min(bw, a.r1 - b0));
  for (int e = threadIdx.x; e < a.r0 * a.d * nbw; e += TM_THREADS) {
    const int row = e / nbw, bb = e - row * nbw;
    const double v = __ldcg(V + size_t(row) * a.r1 + b0 + bb);
    double* p = s.P + row * bw + bb;
    *p = beta == 0.0 ? v : fma(beta, *p, v);
  }
}

// Ap of this CTA's elements from the P of its team.
__device__ void tm_apply(const TeamArgs& a, const TeamSmem& s, int team, int rank) {
  const int r0 = a.r0, r1 = a.r1, w0 = a.w0, w1 = a.w1, d = a.d, bw = a.bw, tid = threadIdx.x;
  const int e0 = rank * a.ew, new_ = max(0, min(a.ew, r1 - e0));
  const int K = w1 * r1, Kp = K + 1;
  const int b0 = rank * bw, nbw = max(0, min(bw, r1 - b0));
  cgrp::cluster_group cl = cgrp::this_cluster();
  for (int q = 0; q < a.rows; ++q) {   // several rows only where a team is one CTA
    const int c = team + q * a.teams;
    const bool live = c < r0;
    __syncthreads();
    if (live) {   // T1[w, t, b]
      // One thread an output, in the order of qtt_cg.cu's stage A: terms that cancel there cancel here.
      // Sums split over lanes cost as much time (a shuffle level is 110 clocks, an fma 64) and took steps from
      // rest (chi = 8) five times further from the oracle.
      const int outs = w0 * d * nbw;
      const double* Lc = s.L + size_t(q) * w0 * r0;
      for (int o = tid; o < outs; o += TM_THREADS) {
        const int bb = o % nbw, wt = o / nbw, t = wt % d, w = wt / d;
        s.T1[wt * bw + bb] = tm_dot<false>(Lc + w * r0, 1, s.P + t * bw + bb, d * bw, r0, 0, 1, true);
      }
    }
    __syncthreads();
    if (live) {   // T2[s, v, b], into every member of the team
      const int outs = d * w1 * nbw;
      for (int o = tid; o < outs; o += TM_THREADS) {
        const int bb = o % nbw, sv = o / nbw, v = sv % w1, s_ = sv / w1;
        double acc = 0.0;
        for (int w = 0; w < w0; ++w)
          for (int t = 0; t < d; ++t)
            acc = fma(s.T1[(w * d + t) * bw + bb], s.W[((w * d + s_) * d + t) * w1 + v], acc);
        const int at = s_ * Kp + v * r1 + b0 + bb;
        if (a.cs == 1) s.T2[at] = acc;
        else
          for (int k = 0; k < a.cs; ++k) cl.map_shared_rank(s.T2, team * a.cs + k)[at] = acc;
      }
    }
    if (a.cs > 1) cl.sync();
    else __syncthreads();
    if (live) {   // Ap[s, e]
      const int outs = d * new_, nl = tm_lanes(outs), l = tid % nl;
      for (int o0 = 0; o0 < outs; o0 += TM_THREADS / nl) {
        const int o = o0 + tid / nl;
        const bool in = o < outs;
        const int oo = in ? o : 0, e = oo % max(new_, 1), s_ = oo / max(new_, 1);
        const double v = a.rres ? tm_dot<false>(s.T2 + s_ * Kp, 1, s.R + size_t(e) * Kp, 1, K, l, nl, in)
                                : tm_dot<true>(s.T2 + s_ * Kp, 1, a.R + size_t(e0 + e) * K, 1, K, l, nl, in);
        if (in && l == 0) s.Ap[(q * d + s_) * a.ew + e] = v;
      }
    }
  }
  __syncthreads();
}

// Sums of f(k, i) over the CTA's elements for k < ns, one warp a quantity, into part[k gridDim.x + block].
template <class F>
__device__ __forceinline__ void tm_sums(double* part, int ns, int nloc, F f) {
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (k < ns) {
    double v = 0.0;
    for (int i = lane; i < nloc; i += 32) v += f(k, i);
    v = tm_warp_sum(v);
    if (lane == 0) part[k * gridDim.x + blockIdx.x] = v;
  }
}

// The grid's sums (the same in every CTA), one warp a quantity.
__device__ void tm_totals(const double* part, int ns, double* tot) {
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31, G = gridDim.x;
  if (k < ns) {
    double v = 0.0;
    for (int i = lane; i < G; i += 32) v += __ldcg(part + k * G + i);
    v = tm_warp_sum(v);
    if (lane == 0) tot[k] = v;
  }
  __syncthreads();
}

__global__ void __launch_bounds__(TM_THREADS) k_cg_team(const __grid_constant__ TeamArgs a) {
  extern __shared__ __align__(16) double tm_sm[];
  const int r0 = a.r0, r1 = a.r1, w0 = a.w0, w1 = a.w1, d = a.d, tid = threadIdx.x;
  const int team = blockIdx.x / a.cs, rank = blockIdx.x % a.cs;
  const int K = w1 * r1, Kp = K + 1, ncap = a.rows * d * a.ew;
  TeamSmem s;
  s.P = tm_sm;
  s.L = s.P + size_t(r0) * d * a.bw;
  s.W = s.L + size_t(a.rows) * w0 * r0;
  s.T1 = s.W + w0 * d * d * w1;
  s.T2 = s.T1 + w0 * d * a.bw;
  s.x = s.T2 + d * Kp;
  s.r = s.x + ncap;
  s.p = s.r + ncap;
  s.Ap = s.p + ncap;
  s.di = s.Ap + ncap;
  s.R = s.di + ncap;
  __shared__ double tot[TM_SUMS];
  __shared__ int err;
  if (tid == 0) err = 0;
  // a CTA's shared memory may be written by its cluster only once the CTA has started
  cgrp::this_cluster().sync();
  const int e0 = rank * a.ew, new_ = max(0, min(a.ew, r1 - e0));
  // operands of the whole solve
  for (int e = tid; e < w0 * d * d * w1; e += TM_THREADS) s.W[e] = __ldg(a.W + e);
  for (int q = 0; q < a.rows; ++q) {
    const int c = team + q * a.teams;
    if (c < r0)
      for (int e = tid; e < w0 * r0; e += TM_THREADS) s.L[size_t(q) * w0 * r0 + e] = __ldg(a.L + size_t(c) * w0 * r0 + e);
  }
  if (a.rres)
    for (int e = tid; e < new_ * K; e += TM_THREADS) s.R[size_t(e / K) * Kp + e % K] = __ldg(a.R + size_t(e0) * K + e);
  // this CTA's elements: i = (q d + s) ew + e; unused places hold zeros
  __syncthreads();
  for (int i = tid; i < ncap; i += TM_THREADS) {
    const int e = i % a.ew, s_ = (i / a.ew) % d, q = i / (a.ew * d), c = team + q * a.teams;
    double x = 0.0, di = 0.0;
    if (c < r0 && e < new_) {
      x = a.xin[(size_t(c) * d + s_) * r1 + e0 + e];
      // the inverse of the local matrix's diagonal, 1 where that is not positive
      double acc = 0.0;
      const double* Re = a.R + size_t(e0 + e) * K + (e0 + e);
      for (int w = 0; w < w0; ++w) {
        double t = 0.0;
        for (int v = 0; v < w1; ++v) t = fma(s.W[((w * d + s_) * d + s_) * w1 + v], __ldg(Re + v * r1), t);
        acc = fma(s.L[(size_t(q) * w0 + w) * r0 + c], t, acc);
      }
      di = acc > 0.0 ? 1.0 / acc : 1.0;
    }
    s.x[i] = x;
    s.di[i] = di;
    s.r[i] = 0.0;
    s.p[i] = 0.0;
    s.Ap[i] = 0.0;
  }
  // r = b - A x, p = z = D r
  tm_direction(a, s, a.xin, 0.0, rank);
  tm_apply(a, s, team, rank);
  for (int i = tid; i < ncap; i += TM_THREADS) {
    const int e = i % a.ew, s_ = (i / a.ew) % d, q = i / (a.ew * d), c = team + q * a.teams;
    if (c < r0 && e < new_) {
      const size_t g = (size_t(c) * d + s_) * r1 + e0 + e;
      const double bv = __ldg(a.b + g), re = bv - s.Ap[i], z = s.di[i] * re;
      s.r[i] = re;
      s.p[i] = z;
      s.Ap[i] = bv;          // for b.b
      a.z[g] = z;
    }
  }
  __syncthreads();
  double* const part0 = a.part;
  double* const part1 = a.part + TM_SUMS * gridDim.x;
  tm_sums(part1, 3, ncap, [&](int k, int i) {
    const double x = k == 0 ? s.Ap[i] : s.r[i];
    return k == 2 ? x * (s.di[i] * x) : x * x;
  });
  tm_sync(a, &err);
  tm_totals(part1, 3, tot);
  const double tol2bb = __ldg(a.tol) * __ldg(a.tol) * tot[0];
  double rr = tot[1], rz = tot[2], beta = 0.0;
  int count = 0;
  for (int it = 0; it < a.iters && rr > tol2bb && rr > 0.0; ++it) {   // the same decisions in every CTA
    tm_direction(a, s, a.z, beta, rank);
    tm_apply(a, s, team, rank);
    tm_sums(part0, 1, ncap, [&](int, int i) { return s.p[i] * s.Ap[i]; });
    tm_sync(a, &err);
    tm_totals(part0, 1, tot);
    const double pap = tot[0];
    if (!(pap > 0.0)) break;
    const double alpha = rz / pap;
    count += 1;
    for (int i = tid; i < ncap; i += TM_THREADS) {
      const int e = i % a.ew, s_ = (i / a.ew) % d, q = i / (a.ew * d), c = team + q * a.teams;
      if (c < r0 && e < new_) {
        const double re = fma(-alpha, s.Ap[i], s.r[i]);
        s.x[i] = fma(alpha, s.p[i], s.x[i]);
        s.r[i] = re;
        a.z[(size_t(c) * d + s_) * r1 + e0 + e] = s.di[i] * re;
      }
    }
    __syncthreads();
    tm_sums(part1, 2, ncap, [&](int k, int i) {
      const double x = s.r[i];
      return k == 1 ? x * (s.di[i] * x) : x * x;
    });
    tm_sync(a, &err);
    tm_totals(part1, 2, tot);
    rr = tot[0];
    beta = tot[1] / rz;
    rz = tot[1];
    for (int i = tid; i < ncap; i += TM_THREADS) s.p[i] = fma(beta, s.p[i], s.di[i] * s.r[i]);
  }
  for (int i = tid; i < ncap; i += TM_THREADS) {
    const int e = i % a.ew, s_ = (i / a.ew) % d, q = i / (a.ew * d), c = team + q * a.teams;
    if (c < r0 && e < new_) a.xout[(size_t(c) * d + s_) * r1 + e0 + e] = s.x[i];
  }
  cgrp::this_cluster().sync();   // no CTA leaves while another may write to its shared memory
  if (blockIdx.x == 0 && tid == 0) {
    if (a.total) {
      if (err) *a.total = TM_POISON;
      else *a.total += count;
    }
    if (a.flops && !err) atomicAdd(a.flops, (count + 1) * a.fpi);
  }
}

struct TeamPlan {
  int cs, teams, bw, ew, rows, rres, grid;
  size_t smem;
};

size_t team_doubles(const TeamPlan& p, int r0, int r1, int w0, int w1, int d) {
  const size_t K = size_t(w1) * r1;
  return size_t(r0) * d * p.bw + size_t(p.rows) * w0 * r0 + size_t(w0) * d * d * w1 + size_t(w0) * d * p.bw + d * (K + 1) +
         5 * size_t(p.rows) * d * p.ew + (p.rres ? size_t(p.ew) * (K + 1) : 0);
}

// Clusters of cs CTAs with that much shared memory that are resident together (cached; the
// occupancy query is a host call of some 10 us).
int team_max_clusters(int cs, size_t smem) {
  static std::mutex mu;
  static std::map<std::pair<int, size_t>, int> known;
  std::lock_guard<std::mutex> lock(mu);
  const std::pair<int, size_t> key(cs, (smem + 8191) / 8192 * 8192);
  auto it = known.find(key);
  if (it != known.end()) return it->second;
  static bool attr = false, attr_ok = false;
  if (!attr) {
    attr = true;
    attr_ok = cudaFuncSetAttribute(k_cg_team, cudaFuncAttributeMaxDynamicSharedMemorySize, int(TM_SMEM)) == cudaSuccess &&
              cudaFuncSetAttribute(k_cg_team, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
  }
  int nclusters = 0;
  if (attr_ok) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(cs));
    cfg.blockDim = dim3(TM_THREADS);
    cfg.dynamicSmemBytes = std::min(key.second, TM_SMEM);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = unsigned(cs);
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&nclusters, k_cg_team, &cfg) != cudaSuccess) nclusters = 0;
  }
  cudaGetLastError();
  known[key] = nclusters;
  return nclusters;
}

// One cluster up to r0 r1 = 256.  Poisson solves on 10 bits, against the cooperative kernel of qtt_cg.cu
// (same iterations): all bonds <= 8 13.0 -> 9.5 ms (210 iterations, 4 sweeps), <= 12 11.4 -> 8.3 ms, <= 16
// 10.3 -> 7.7 ms.  Larger sites want more than 16 CTAs and stay with the cooperative kernels.
bool cg_team_plan(int r0, int r1, int w0, int w1, int d, TeamPlan& p) {
  if (!(r0 >= 1 && r1 >= 1 && r0 * int64_t(r1) <= TM_ELEMS && w0 >= 1 && w1 >= 1 && w0 <= 16 && w1 <= 16 && d >= 1 && d <= 4))
    return false;
  p.teams = std::min(r0, TM_CLUSTER);
  p.cs = 1;
  while (p.teams * p.cs * 2 <= TM_CLUSTER && p.cs * 2 <= r1) p.cs *= 2;
  p.rows = (r0 + p.teams - 1) / p.teams;
  p.bw = p.ew = (r1 + p.cs - 1) / p.cs;
  p.grid = p.teams * p.cs;
  p.rres = 1;
  p.smem = team_doubles(p, r0, r1, w0, w1, d) * sizeof(double);
  if (p.smem > TM_SMEM) {
    p.rres = 0;
    p.smem = team_doubles(p, r0, r1, w0, w1, d) * sizeof(double);
    if (p.smem > TM_SMEM) return false;
  }
  return team_max_clusters(p.grid, p.smem) >= 1;
}

}  // namespace

bool cg_team_fits(int r0, int r1, int w0, int w1, int d) {
  TeamPlan p;
  return cg_team_plan(r0, r1, w0, w1, d, p);
}

void cg_team(Ctx& c, const double* L, const double* W, const double* R, const double* b, const double* xin, double* xout,
             int r0, int r1, int w0, int w1, int d, int iters, const double* tol_dev, int* total_dev) {
  TeamPlan p;
  QTT_CHECK_ARG(cg_team_plan(r0, r1, w0, w1, d, p), "cg_team: shape outside the supported range");
  DBuf zbuf(&c, size_t(r0) * d * r1), part(&c, size_t(2 * TM_SUMS) * p.grid);
  TeamArgs a;
  a.r0 = r0; a.r1 = r1; a.w0 = w0; a.w1 = w1; a.d = d; a.iters = iters;
  a.cs = p.cs; a.teams = p.teams; a.bw = p.bw; a.ew = p.ew; a.rows = p.rows; a.rres = p.rres;
  a.tol = tol_dev;
  a.L = L; a.W = W; a.R = R; a.b = b; a.xin = xin; a.xout = xout;
  a.z = zbuf.p; a.part = part.p;
  a.limit_ns = c.root->wait_ns;
  a.total = total_dev;
  a.flops = c.root->prof.on ? c.root->prof.dev_flops : nullptr;
  a.fpi = 2.0 * (double(r0) * w0 * r0 * d * r1 + double(r0) * d * w0 * d * w1 * r1 + double(r0) * d * w1 * r1 * r1);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(p.grid));
  cfg.blockDim = dim3(TM_THREADS);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = c.stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = unsigned(p.grid);
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;   // a cluster is resident as a whole: no cooperative launch
  ProfScope ps(c, KC_CG);
  QTT_CUDA(cudaLaunchKernelEx(&cfg, k_cg_team, a));
  after_launch(c, "cg_team");
}

}  // namespace qtt

// Eigenpairs of the density matrices of the roundings (symmetric positive semidefinite, order up
// to 128): a single-CTA start in FP32 and an FP64 refinement as one cooperative grid, a level for
// every eight decades of the spectrum.
//
// Start (k_psd_start, one CTA): the diagonally pivoted Cholesky factor L of the scaled matrix in
// two-float arithmetic (48 bits), then one-sided Jacobi on the columns of L in FP32 (Veselic and
// Hari, Numer. Math. 56, 1989): the columns converge to sigma_j u_j, so the eigenvectors come out
// without accumulating rotations, and because the pivoted factor is graded every column is known
// relative to its own length, eight decades down the spectrum, not to ||S||.  The factor stops at the
// pivot floor; the vectors below it (the next level's, or null vectors) are a Householder basis of the
// orthogonal complement.
// Refinement (k_psd_refine): Newton-Schulz and Ogita-Aishima iterations (Ogita and Aishima, Japan
// J. Indust. Appl. Math. 35, 2018) until the next correction across the cut would be below rounding (at
// most eight; all eight where the cut lies among eigenvalues of pure rounding, whose corrections do not shrink),
// products of 8 x 8 tiles dealt to the CTAs, grid
// barriers (bounded, as in qtt_cg.cu) between them.  With a factor F (S = F^T F) X^T S X is formed
// as (F X)^T (F X), which keeps the tail on its own scale, and levels follow down to 1e-24.
//
// What bounds it: the start is a chain of n - 1 rotation rounds a sweep, each about 0.2 us of
// shared-memory and shuffle latency on one SM; the refinement is bound by the FP64 pipe at n = 128
// (2 FMA a clock and SM: a product of order 128 takes 3.4 us of the whole chip) and by the grid
// barrier (1.3 us) below n = 64.  The path that it replaces for these matrices (two-sided FP32
// Jacobi of 1.5 us a round, levels three decades apart, some 35 launches a level; qtt_linalg.cu,
// which stays for indefinite matrices and orders above 128) is measured against it at eigh_psd_fits.
#include <algorithm>

#include "qtt_algebra.h"

namespace qtt {

namespace {

constexpr int PS_MAX_N = 128;
constexpr int PS_THREADS = 512;
constexpr int PS_MAX_SWEEPS = 14;
constexpr float PS_FLOOR = 1e-13f;      // pivots below are treated as zero (entries of the scaled matrix are < 2)
constexpr float PS_ROT = 3e-7f;         // a pair closer to orthogonal is left alone
constexpr float PS_DONE = 1e-3f;        // a sweep that met no larger cosine is the last (quadratic convergence)

// Barrier and result record of one eigenproblem (device memory, set up by its start kernels).
struct PsdState {
  unsigned int count;      // arrivals at the level's barriers; top bit: a CTA gave up waiting
  unsigned int left;       // CTAs that left the level because of that
  unsigned long long limit_ns;
  int t0, need;            // the next level's tail block and whether it is taken
  int e;                   // the matrix is worked on as S 2^-e
  int pad;
  double anorm;            // ||S 2^-e||_F, from level 0's refinement
};

__device__ __forceinline__ unsigned long long f2_fma(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long f2_mul(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long f2_set(float v) {
  unsigned long long d;
  asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(v));
  return d;
}
__device__ __forceinline__ float fast_rsqrt(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float fast_rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float f2_sum(unsigned long long a) {
  float x, y;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a));
  return x + y;
}

// Columns are rotated in blocks of four: sixteen lanes hold the eight columns of a block pair in
// registers (TT x 4 rows a lane, 16-byte shared-memory accesses) and rotate each column of one
// block with each of the other in four rounds of four disjoint pairs; round-robin over the blocks.
// Rotating every pair straight from shared memory moves all columns through it n - 1 times a
// sweep (128 KB a round at n = 128: 1024 clocks, which bounded it at about 0.8 us a round); blocks
// of four need a quarter of that.  The four dot products of a round are summed over the lanes
// by a reduce-scatter, so each lane forms one pair's rotation and hands it to the others.
template <int TT>
struct PsCols {
  ulonglong2 v[8][TT];   // columns 0-3: first block, 4-7: second
  float nrm[8];
};

// Rotate the pairs (P[k], Q[k]), k = 0..3, of the eight columns; returns the largest cosine met.
template <int TT, int P0, int Q0, int P1, int Q1, int P2, int Q2, int P3, int Q3>
__device__ __forceinline__ float ps_rotate4(PsCols<TT>& c, int lane) {
  constexpr int P[4] = {P0, P1, P2, P3}, Q[4] = {Q0, Q1, Q2, Q3};
  float g[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    unsigned long long a = f2_mul(c.v[P[k]][0].x, c.v[Q[k]][0].x);
    a = f2_fma(c.v[P[k]][0].y, c.v[Q[k]][0].y, a);
#pragma unroll
    for (int t = 1; t < TT; ++t) {
      a = f2_fma(c.v[P[k]][t].x, c.v[Q[k]][t].x, a);
      a = f2_fma(c.v[P[k]][t].y, c.v[Q[k]][t].y, a);
    }
    g[k] = f2_sum(a);
  }
  // lanes with (bit 0, bit 1) = (k & 1, k >> 1) end with the sum of pair k
  const bool b0 = lane & 1, b1 = lane & 2;
  float u0 = b0 ? g[1] : g[0], u1 = b0 ? g[3] : g[2];
  u0 += __shfl_xor_sync(0xffffffffu, b0 ? g[0] : g[1], 1);
  u1 += __shfl_xor_sync(0xffffffffu, b0 ? g[2] : g[3], 1);
  float gamma = b1 ? u1 : u0;
  gamma += __shfl_xor_sync(0xffffffffu, b1 ? u0 : u1, 2);
  gamma += __shfl_xor_sync(0xffffffffu, gamma, 4);
  gamma += __shfl_xor_sync(0xffffffffu, gamma, 8);
  const float alpha = b1 ? (b0 ? c.nrm[P3] : c.nrm[P2]) : (b0 ? c.nrm[P1] : c.nrm[P0]);
  const float beta = b1 ? (b0 ? c.nrm[Q3] : c.nrm[Q2]) : (b0 ? c.nrm[Q1] : c.nrm[Q0]);
  // t = tan(theta) = sign(delta gamma) |2 gamma| / (|delta| + sqrt(delta^2 + 4 gamma^2))
  const float cosv = fabsf(gamma) * fast_rsqrt(alpha * beta);
  const bool rot = cosv > PS_ROT;              // false for the zero columns of the padding
  const float del = beta - alpha, g2 = gamma + gamma;
  const float h2 = fmaf(del, del, g2 * g2);
  const float h = h2 * fast_rsqrt(h2);
  const float tt = g2 * fast_rcp(fabsf(del) + h);
  const float t = rot ? (del < 0.f ? -tt : tt) : 0.f;
  const float cs = fast_rsqrt(fmaf(t, t, 1.f)), tg = rot ? t * gamma : 0.f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float tk = __shfl_sync(0xffffffffu, t, k, 16), ck = __shfl_sync(0xffffffffu, cs, k, 16);
    const float gk = __shfl_sync(0xffffffffu, tg, k, 16), sk = tk * ck;
    c.nrm[P[k]] -= gk;
    c.nrm[Q[k]] += gk;
    const unsigned long long c2 = f2_set(ck), s2 = f2_set(sk), m2 = f2_set(-sk);
#pragma unroll
    for (int r = 0; r < TT; ++r) {
      const ulonglong2 x = c.v[P[k]][r], y = c.v[Q[k]][r];
      c.v[P[k]][r].x = f2_fma(c2, x.x, f2_mul(m2, y.x));
      c.v[P[k]][r].y = f2_fma(c2, x.y, f2_mul(m2, y.y));
      c.v[Q[k]][r].x = f2_fma(s2, x.x, f2_mul(c2, y.x));
      c.v[Q[k]][r].y = f2_fma(s2, x.y, f2_mul(c2, y.y));
    }
  }
  return rot ? cosv : 0.f;
}

// One sweep over the nb blocks of four columns (nb even; leading dimension ld floats, TT x 64 rows).
// nrm2: squared column norms, formed anew at the start of the sweep and updated with the rotations.
template <int TT>
__device__ void ps_sweep(float* A, int ld, int nb, float* nrm2, unsigned int* worst) {
  const int tid = threadIdx.x, g = tid >> 4, l = tid & 15;
  for (int r = 0; r < nb - 1; ++r) {
    const bool act = g < nb / 2;
    if (__any_sync(0xffffffffu, act)) {
      int p = 0, q = 0;
      if (act) {
        if (g == 0) { p = r; q = nb - 1; }
        else {
          p = r + g; if (p >= nb - 1) p -= nb - 1;
          q = r - g; if (q < 0) q += nb - 1;
        }
        if (p > q) { const int t = p; p = q; q = t; }
      }
      PsCols<TT> c;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int col = 4 * (k < 4 ? p : q) + (k & 3);
        c.nrm[k] = act ? nrm2[col] : 0.f;
#pragma unroll
        for (int t = 0; t < TT; ++t)
          c.v[k][t] = act ? *reinterpret_cast<const ulonglong2*>(A + size_t(col) * ld + 64 * t + 4 * l) : make_ulonglong2(0ull, 0ull);
      }
      float w = 0.f;
      if (r == 0) {   // the pairs within the blocks, once a sweep
        w = fmaxf(w, ps_rotate4<TT, 0, 1, 2, 3, 4, 5, 6, 7>(c, l));
        w = fmaxf(w, ps_rotate4<TT, 0, 2, 1, 3, 4, 6, 5, 7>(c, l));
        w = fmaxf(w, ps_rotate4<TT, 0, 3, 1, 2, 4, 7, 5, 6>(c, l));
      }
      w = fmaxf(w, ps_rotate4<TT, 0, 4, 1, 5, 2, 6, 3, 7>(c, l));
      w = fmaxf(w, ps_rotate4<TT, 0, 5, 1, 6, 2, 7, 3, 4>(c, l));
      w = fmaxf(w, ps_rotate4<TT, 0, 6, 1, 7, 2, 4, 3, 5>(c, l));
      w = fmaxf(w, ps_rotate4<TT, 0, 7, 1, 4, 2, 5, 3, 6>(c, l));
      if (act) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int col = 4 * (k < 4 ? p : q) + (k & 3);
          if (l == k) nrm2[col] = c.nrm[k];
#pragma unroll
          for (int t = 0; t < TT; ++t) *reinterpret_cast<ulonglong2*>(A + size_t(col) * ld + 64 * t + 4 * l) = c.v[k][t];
        }
        if (l < 4 && w > 0.f) atomicMax(worst, __float_as_uint(fminf(w, 2.f)));
      }
    }
    __syncthreads();
  }
}

// nrm2[c] = |column c|^2, one warp a column.
__device__ void ps_norms(const float* A, int ld, int rows, int cols, float* nrm2) {
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int c = ty; c < cols; c += PS_THREADS / 32) {
    float s = 0.f;
    for (int i = tx; i < rows; i += 32) s = fmaf(A[size_t(c) * ld + i], A[size_t(c) * ld + i], s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (tx == 0) nrm2[c] = s;
  }
}

// Shared memory of the start (floats): A, the factor's columns (a multiple of eight, ld each); B, their
// low parts; the matrix as packed lower triangles of high and low parts; diagonals, norms, order.
__host__ __device__ constexpr int ps_ld(int n) { return (n + 63) / 64 * 64 + 4; }
__host__ __device__ constexpr int ps_cols(int n) { return (n + 7) / 8 * 8; }
__host__ __device__ constexpr size_t ps_smem(int n) {
  return (2 * size_t(ps_cols(n)) * ps_ld(n) + size_t(n) * (n + 1) + 6 * PS_MAX_N) * sizeof(float);
}
__device__ __forceinline__ int ps_tri(int i, int k) { return i >= k ? i * (i + 1) / 2 + k : k * (k + 1) / 2 + i; }

// (h, l) -= (ah, al) (bh, bl) in two-float arithmetic (the product's error and the difference's error
// kept; about 2^-46 relative).
__device__ __forceinline__ void ff_submul(float& h, float& l, float ah, float al, float bh, float bl) {
  const float p = __fmul_rn(ah, bh);
  float e = __fmaf_rn(ah, bh, -p);
  e = __fmaf_rn(ah, bl, e);
  e = __fmaf_rn(al, bh, e);
  const float s = __fsub_rn(h, p);
  const float z = __fsub_rn(s, h);
  const float er = __fsub_rn(__fsub_rn(h, __fsub_rn(s, z)), __fadd_rn(p, z));
  const float lo = __fadd_rn(l, __fsub_rn(er, e));
  h = __fadd_rn(s, lo);
  l = __fsub_rn(lo, __fsub_rn(h, s));
}
__device__ __forceinline__ void ff_add(float& h, float& l, float bh, float bl) {
  const float s = __fadd_rn(h, bh);
  const float z = __fsub_rn(s, h);
  const float er = __fadd_rn(__fsub_rn(h, __fsub_rn(s, z)), __fsub_rn(bh, z));
  const float lo = __fadd_rn(__fadd_rn(l, bl), er);
  h = __fadd_rn(s, lo);
  l = __fsub_rn(lo, __fsub_rn(h, s));
}

// Start of one level.  level 0: the n x n matrix S (row-major; scaled copy to Ssc, state set up);
// else the tail block S[t0:, t0:] (order nfull - t0) of the sorted X^T S X, when st->need.  Xout
// (order x order, row-major): the start's eigenvectors, columns by decreasing eigenvalue.
__global__ void __launch_bounds__(PS_THREADS) k_psd_start(int nfull, const double* __restrict__ S, int even,
                                                          double* __restrict__ Ssc, double* __restrict__ Xout,
                                                          PsdState* st, int level, unsigned long long limit_ns) {
  extern __shared__ __align__(16) float ps_sm[];
  if (level > 0 && st->need == 0) return;
  const int t0 = level > 0 ? st->t0 : 0;
  const int n = nfull - t0, ld = ps_ld(n);
  const int nc = ps_cols(n);
  float* A = ps_sm;
  float* B = A + size_t(nc) * ld;
  float* Sh = B + size_t(nc) * ld;
  float* Sl = Sh + n * (n + 1) / 2;
  float* dh = Sl + n * (n + 1) / 2;      // diagonal of what is left (two floats)
  float* dl = dh + PS_MAX_N;
  float* nrm2 = dl + PS_MAX_N;
  float* vd = nrm2 + PS_MAX_N;
  float* vi = vd + PS_MAX_N;
  int* order = reinterpret_cast<int*>(vi + PS_MAX_N);
  __shared__ double red[PS_THREADS / 32];
  __shared__ int es;
  __shared__ unsigned int worst;
  const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
  // scale exponent: largest entry into [1, 2) ([1, 4) for an even exponent)
  double mx = 0.0;
  for (int e = tid; e < n * n; e += PS_THREADS) {
    const double v = fabs(S[size_t(e / n + t0) * nfull + (e % n + t0)]);
    mx = v > mx ? v : mx;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double v = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = v > mx ? v : mx;
  }
  if (tx == 0) red[ty] = mx;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int w = 0; w < PS_THREADS / 32; ++w) t = red[w] > t ? red[w] : t;
    int e = (t > 0.0 && isfinite(t)) ? ilogb(t) : 0;
    if (even && (e & 1)) e -= 1;
    es = e;
  }
  __syncthreads();
  const int e0 = es;
  for (int e = tid; e < n * n; e += PS_THREADS) {
    const int i = e / n, k = e % n;
    const double v = ldexp(S[size_t(i + t0) * nfull + (k + t0)], -e0);
    if (level == 0) Ssc[size_t(i) * nfull + k] = v;
    const float h = float(v), lo = float(v - double(h));
    if (k <= i) {
      Sh[ps_tri(i, k)] = h;
      Sl[ps_tri(i, k)] = lo;
      if (i == k) { dh[i] = h; dl[i] = lo; }
    }
  }
  for (int i = n + tid; i < PS_MAX_N; i += PS_THREADS) dh[i] = 0.f;
  for (int e = tid; e < nc * ld; e += PS_THREADS) A[e] = 0.f;
  __syncthreads();
  if (tid == 0) {
    if (level == 0) st->e = e0;
    st->limit_ns = limit_ns;
    st->count = 0;
    st->left = 0;
  }
  // Pivoted Cholesky, left-looking: the pivot's column is formed when it is chosen (four lanes a
  // row share the sum over the earlier columns), only the diagonal is kept up to date.  Every
  // warp finds the same pivot; a used row's diagonal is zero.
  int j = 0;
  for (; j < n; ++j) {
    unsigned int key = 0u;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int i = tx + 32 * t;
      const float d = dh[i];
      if (d > PS_FLOOR) key = max(key, (__float_as_uint(d) & ~127u) | unsigned(127 - i));
    }
    key = __reduce_max_sync(0xffffffffu, key);
    if (key == 0u) break;
    const int p = 127 - int(key & 127u);
    const int i = tid >> 2, q = tid & 3;
    const float ph = dh[p], pl = dl[p];
    float h = 0.f, l = 0.f;
    const bool live = i < n && dh[i] > 0.f;
    if (live) {
      if (q == 0) {
        h = Sh[ps_tri(i, p)];
        l = Sl[ps_tri(i, p)];
      }
      for (int k = q; k < j; k += 4)
        ff_submul(h, l, A[size_t(k) * ld + i], B[size_t(k) * ld + i], A[size_t(k) * ld + p], B[size_t(k) * ld + p]);
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      const float oh = __shfl_xor_sync(0xffffffffu, h, o), ol = __shfl_xor_sync(0xffffffffu, l, o);
      ff_add(h, l, oh, ol);
    }
    // 1 / sqrt(pivot) to two floats: r + r (1 - d r^2) / 2
    const float r = fast_rsqrt(ph);
    const float r2 = __fmul_rn(r, r), r2e = __fmaf_rn(r, r, -r2);
    const float q1 = __fmul_rn(ph, r2);
    float res = __fsub_rn(1.f, q1);
    res = __fsub_rn(res, __fmaf_rn(ph, r2, -q1));
    res = __fsub_rn(res, __fmaf_rn(ph, r2e, __fmul_rn(pl, r2)));
    const float rl = __fmul_rn(__fmul_rn(0.5f, r), res);
    // column entry (h, l) (r, rl)
    const float ch = __fmul_rn(h, r);
    float cl = __fmaf_rn(h, r, -ch);
    cl = __fmaf_rn(h, rl, __fmaf_rn(l, r, cl));
    const float lh = __fadd_rn(ch, cl), ll = __fsub_rn(cl, __fsub_rn(lh, ch));
    __syncthreads();                                    // every read of the diagonal is done
    if (live && q == 0) {
      A[size_t(j) * ld + i] = lh;
      B[size_t(j) * ld + i] = ll;
      float a = dh[i], b = dl[i];
      ff_submul(a, b, lh, ll, lh, ll);
      dh[i] = i == p ? 0.f : fmaxf(a, 0.f);             // a row rounded down to zero is never chosen
      dl[i] = b;
    }
    __syncthreads();
  }
  // one-sided Jacobi
  const int rk = j, nb = ps_cols(rk) / 4;
  for (int sweep = 0; sweep < PS_MAX_SWEEPS && nb > 0; ++sweep) {
    if (tid == 0) worst = 0u;
    ps_norms(A, ld, n, 4 * nb, nrm2);
    __syncthreads();
    if (n <= 64) ps_sweep<1>(A, ld, nb, nrm2, &worst);
    else ps_sweep<2>(A, ld, nb, nrm2, &worst);
    const float wv = __uint_as_float(worst);
    __syncthreads();
    if (!(wv > PS_DONE)) break;
  }
  // lengths, order; the normalised columns to Xout and to B
  ps_norms(A, ld, n, rk, nrm2);
  __syncthreads();
  for (int c = tid; c < rk; c += PS_THREADS) {
    const unsigned int kc = __float_as_uint(nrm2[c]);   // lengths are not negative: ordered as integers
    int rank = 0;
    for (int o = 0; o < rk; ++o) {
      const unsigned int ko = __float_as_uint(nrm2[o]);
      rank += (ko > kc || (ko == kc && o < c)) ? 1 : 0;
    }
    order[rank] = c;
  }
  __syncthreads();
  for (int e = tid; e < n * rk; e += PS_THREADS) {
    const int k = e / n, i = e - k * n, c = order[k];
    const float v = A[size_t(c) * ld + i] * rsqrtf(nrm2[c]);
    B[size_t(k) * ld + i] = v;
    Xout[size_t(i) * n + k] = double(v);
  }
  if (rk == n) return;
  // The orthogonal complement: Householder reflectors of the rk nearly orthonormal columns in B
  // (reflector k: rows below k of its column, vd[k] on the diagonal, factor vi[k]), then
  // columns rk .. n - 1 of their product, each by one warp.
  __syncthreads();
  for (int k = 0; k < rk; ++k) {
    float v[4], sg = 0.f, al = 0.f;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int i = tx + 32 * t;
      const float x = i < n ? B[size_t(k) * ld + i] : 0.f;
      v[t] = i > k ? x : 0.f;
      if (i == k) al = x;
      sg = fmaf(v[t], v[t], sg);
    }
    for (int o = 16; o > 0; o >>= 1) sg += __shfl_xor_sync(0xffffffffu, sg, o);
    al = __shfl_sync(0xffffffffu, al, k & 31);
    const float q = fmaf(al, al, sg), nr = q > 0.f ? q * fast_rsqrt(q) : 0.f;
    const float v0 = al >= 0.f ? al + nr : al - nr;
    const float inv = nr > 0.f ? fast_rcp(nr * (nr + fabsf(al))) : 0.f;
    if (tid == 0) { vd[k] = v0; vi[k] = inv; }
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (tx + 32 * t == k) v[t] = v0;
    for (int c0 = k + 1 + ty; c0 < rk; c0 += 4 * (PS_THREADS / 32)) {   // four columns a warp at a time
      float y[4][4], w[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int c = c0 + m * (PS_THREADS / 32);
        w[m] = 0.f;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int i = tx + 32 * t;
          y[m][t] = (c < rk && i < n) ? B[size_t(c) * ld + i] : 0.f;
          w[m] = fmaf(v[t], y[m][t], w[m]);
        }
      }
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int m = 0; m < 4; ++m) w[m] += __shfl_xor_sync(0xffffffffu, w[m], o);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int c = c0 + m * (PS_THREADS / 32);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int i = tx + 32 * t;
          if (c < rk && i < n) B[size_t(c) * ld + i] = fmaf(-w[m] * inv, v[t], y[m][t]);
        }
      }
    }
    __syncthreads();
  }
  for (int c0 = rk + ty; c0 < n; c0 += 4 * (PS_THREADS / 32)) {   // four columns a warp at a time
    float y[4][4];
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int t = 0; t < 4; ++t) y[m][t] = (tx + 32 * t == c0 + m * (PS_THREADS / 32)) ? 1.f : 0.f;
    for (int k = rk - 1; k >= 0; --k) {
      const float* x = B + size_t(k) * ld;
      const float v0 = vd[k], inv = vi[k];
      float v[4], w[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int i = tx + 32 * t;
        v[t] = (i < n && i > k) ? x[i] : (i == k ? v0 : 0.f);
#pragma unroll
        for (int m = 0; m < 4; ++m) w[m] = fmaf(v[t], y[m][t], w[m]);
      }
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int m = 0; m < 4; ++m) w[m] += __shfl_xor_sync(0xffffffffu, w[m], o);
#pragma unroll
      for (int m = 0; m < 4; ++m)
#pragma unroll
        for (int t = 0; t < 4; ++t) y[m][t] = fmaf(-w[m] * inv, v[t], y[m][t]);
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int c = c0 + m * (PS_THREADS / 32);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int i = tx + 32 * t;
        if (c < n && i < n) Xout[size_t(i) * n + c] = double(y[m][t]);
      }
    }
  }
}

// ------------------------------------------------------------------ refinement

constexpr int PR_THREADS = 256;
constexpr int PR_T = 8;                 // output tile
constexpr int PR_MAX_IT = 8;            // Ogita-Aishima iterations of one level at most
constexpr float PR_STOP = 1e-14f;        // predicted size of the next correction across the cut
constexpr double PR_STEP = 1e-2;         // largest correction within one side of the cut

struct PsdArgs {
  int n, m, keep, level;
  const double* S;      // scaled matrix (used without a factor)
  const double* F;      // scaled factor (m x n) or null
  const double* Y;      // the start's vectors: X itself at level 0, the tail block's basis after
  double* V;            // in/out: eigenvectors, columns by decreasing eigenvalue
  double* w;            // eigenvalues (unscaled)
  double* lam;          // eigenvalues of the scaled matrix, sorted
  double *X0, *X1, *G, *B, *SX, *E, *SXs;
  double* part;         // 4 x gridDim.x: partial sums of squares of X^T X - I, of the off-diagonal X^T S X, of
                        // its pairs with the block, of S
  float* big;           // gridDim.x: largest correction
  double tau_next;      // threshold of the next level (0: none)
  PsdState* st;
};

__device__ __forceinline__ unsigned int pr_ld_acquire(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long pr_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid barrier on a monotonic arrival counter, bounded by the context's wait limit (see qtt_cg.cu).  A CTA
// gives up by a compare-and-swap on a count that is not complete yet, so that the last barrier is passed by
// every CTA or by none: a level that ran out of time has not touched what it started from.
constexpr unsigned int PR_GAVE_UP = 1u << 31;
struct PsdGrid {
  int G, b;      // CTAs that share the level, this CTA's index among them
};
__device__ bool pr_sync(PsdState* st, const PsdGrid& g, unsigned int& target, int* flag) {
  if (g.G == 1) {
    __threadfence();
    __syncthreads();
    return true;
  }
  target += g.G;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(&st->count), "r"(1u) : "memory");
    const unsigned long long t0 = pr_ns(), limit = st->limit_ns;
    const unsigned int mask = limit < 100000ull ? 0u : 255u;
    unsigned int spins = 0, v;
    while ((v = pr_ld_acquire(&st->count)) < target) {
      if ((++spins & mask) == 0u && pr_ns() - t0 > limit && atomicCAS(&st->count, v, v | PR_GAVE_UP) == v) v |= PR_GAVE_UP;
      if (v & PR_GAVE_UP) break;
    }
    __threadfence();
    *flag = (v & PR_GAVE_UP) != 0u;
  }
  __syncthreads();
  return *flag == 0;
}

// acc = sum_k A(i0 + i, k) B(k, j0 + j) over K for this thread's output (o = tid / 4: i = o / 8,
// j = o % 8), four lanes a piece; A is read as A[k lda + i] (acol) or A[i lda + k].  Values written
// by other CTAs of the launch are read through L2.  Ends with a CTA barrier.
__device__ double pr_tile(const double* A, int lda, bool acol, int i0, int I, const double* B, int ldb, int j0, int J,
                          int K, double* sA, double* sB) {
  const int tid = threadIdx.x;
  const int ldk = K + 2;
  if (acol) {
    for (int e = tid; e < K * PR_T; e += PR_THREADS) {
      const int k = e >> 3, i = e & 7;
      sA[i * ldk + k] = (i0 + i < I) ? __ldcg(A + size_t(k) * lda + i0 + i) : 0.0;
    }
  } else {
    for (int i = tid >> 5; i < PR_T; i += PR_THREADS / 32)
      for (int k = tid & 31; k < K; k += 32) sA[i * ldk + k] = (i0 + i < I) ? __ldcg(A + size_t(i0 + i) * lda + k) : 0.0;
  }
  for (int e = tid; e < K * PR_T; e += PR_THREADS) {
    const int k = e >> 3, j = e & 7;
    sB[e] = (j0 + j < J) ? __ldcg(B + size_t(k) * ldb + j0 + j) : 0.0;
  }
  __syncthreads();
  const int o = tid >> 2, l = tid & 3, i = o >> 3, j = o & 7;
  const double* a = sA + i * ldk;
  const double* b = sB + j;
  double s0 = 0.0, s1 = 0.0;
  int k = l;
  for (; k + 4 < K; k += 8) {
    s0 = fma(a[k], b[k * PR_T], s0);
    s1 = fma(a[k + 4], b[(k + 4) * PR_T], s1);
  }
  if (k < K) s0 = fma(a[k], b[k * PR_T], s0);
  double s = s0 + s1;
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  __syncthreads();
  return s;
}

// Sums over the CTA of v0 and v1, held by the lanes l = tid % 4 = 0, to out0[0] and out1[0]; red: 16 doubles, not
// used again before the next CTA barrier.  Both go through the same additions, on lanes l = 0 and 1.
__device__ __forceinline__ void pr_block_pair(double v0, double v1, double* red, double* out0, double* out1) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, l = lane & 3;
  const double up = __shfl_up_sync(0xffffffffu, v1, 1);
  double v = l == 0 ? v0 : l == 1 ? up : 0.0;
  for (int o = 16; o > 2; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane < 2) red[2 * w + lane] = v;
  __syncthreads();
  if (w == 0) {
    v = lane < 2 * (PR_THREADS / 32) ? red[lane] : 0.0;
    for (int o = PR_THREADS / 32; o > 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) *out0 = v;
    if (lane == 1 && out1) *out1 = v;
  }
}

// Order-preserving integer key of a double, NaN below everything.
__device__ __forceinline__ long long pr_key(double v) {
  if (isnan(v)) return -0x7fffffffffffffffll - 1;
  const long long b = __double_as_longlong(v);
  return b < 0 ? (b ^ 0x7fffffffffffffffll) : b;
}

// Symmetric product P = U^T W (both K x n, row-major; the upper tiles, mirrored) and, when T is
// given, T = L R with L (M x n, row-major) and R (n x n): the tiles of both dealt to the CTAs.
// Sum of squares of (delta_ij - P_ij) (of_identity) or of the off-diagonal P_ij and, of the latter, (tail) of those
// with a column at t0 or beyond; in FP64, as couplings of the deep levels square to below FP32's range.  On
// the lanes tid % 4 = 0.
__device__ double pr_products(const PsdGrid& g, int n, const double* U, const double* W, int K, double* P,
                             bool of_identity, const double* L, const double* R, int M, double* T, int t0, double& tail,
                             double* sA, double* sB) {
  const int nt = (n + PR_T - 1) / PR_T, sym = nt * (nt + 1) / 2, mt = T ? (M + PR_T - 1) / PR_T : 0;
  double diag = 0.0, off = 0.0, offt = 0.0;
  const int tid = threadIdx.x, l = tid & 3, oi = (tid >> 2) >> 3, oj = (tid >> 2) & 7;
  for (int t = g.b; t < sym + mt * nt; t += g.G) {
    if (t < sym) {
      int a = 0, r = t;
      while (r >= nt - a) { r -= nt - a; ++a; }
      const int b = a + r, i = a * PR_T + oi, j = b * PR_T + oj;
      const double s = pr_tile(U, n, true, a * PR_T, n, W, n, b * PR_T, n, K, sA, sB);
      if (l == 0 && i < n && j < n && i <= j) {
        P[size_t(i) * n + j] = s;
        if (i != j) P[size_t(j) * n + i] = s;
        if (i != j) {
          off = fma(s, s, off);
          if (t0 > 0 && j >= t0) offt = fma(s, s, offt);
        } else if (of_identity) {
          diag = fma(1.0 - s, 1.0 - s, diag);
        }
      }
    } else {
      const int q = t - sym, a = q / nt, b = q % nt, i = a * PR_T + oi, j = b * PR_T + oj;
      const double s = pr_tile(L, n, false, a * PR_T, M, R, n, b * PR_T, n, n, sA, sB);
      if (l == 0 && i < M && j < n) T[size_t(i) * n + j] = s;
    }
  }
  tail = 2.0 * (t0 > 0 ? offt : off);
  return fma(2.0, off, diag);
}

// Xo[:, col(j)] = X + X E (mode 0), X (3 I - E) / 2 (mode 1), X E (mode 2); rank: column map or null.
__device__ void pr_update(const PsdGrid& g, int n, const double* X, const double* E, double* Xo, int mode,
                          const int* rank, double* sA, double* sB) {
  const int nt = (n + PR_T - 1) / PR_T;
  const int tid = threadIdx.x, l = tid & 3, oi = (tid >> 2) >> 3, oj = (tid >> 2) & 7;
  for (int t = g.b; t < nt * nt; t += g.G) {
    const int a = t / nt, b = t % nt, i = a * PR_T + oi, j = b * PR_T + oj;
    double s = pr_tile(X, n, false, a * PR_T, n, E, n, b * PR_T, n, n, sA, sB);
    if (l == 0 && i < n && j < n) {
      const double x = mode == 2 ? 0.0 : __ldcg(X + size_t(i) * n + j);
      s = mode == 0 ? x + s : mode == 1 ? fma(-0.5, s, 1.5 * x) : s;
      Xo[size_t(i) * n + (rank ? rank[j] : j)] = s;
    }
  }
}

// One level by the CTAs of g; false, with V, w, lam and SXs as they were, if a wait ran out.
__device__ __forceinline__ bool psd_level(const PsdArgs& a, const PsdGrid& g) {
  extern __shared__ __align__(16) double pr_sm[];
  PsdState* st = a.st;
  const int n = a.n, tid = threadIdx.x, G = g.G;
  const int Kmax = max(n, a.m);
  double* sA = pr_sm;
  double* sB = sA + PR_T * (Kmax + 2);
  double* sl = sB + PR_T * Kmax;            // n eigenvalues
  int* rank = reinterpret_cast<int*>(sl + n);
  __shared__ float redf[PR_THREADS / 32];
  __shared__ double red[2 * (PR_THREADS / 32)], norms[4], delta_s, delta_t;
  __shared__ float tail_s;
  __shared__ float slf[PS_MAX_N];
  __shared__ int flag;
  unsigned int target = 0;
  const int t0 = a.level > 0 ? st->t0 : 0;
  double unused;
  double* X = a.X0;
  double* Xn = a.X1;
  bool ok = true;
  auto swap = [&]() { double* t = X; X = Xn; Xn = t; };
  // eigenvalue estimates of the current X from G = X^T X and SX, and their descending ranks
  auto lambda = [&]() {
    for (int i = tid; i < n; i += PR_THREADS) {
      sl[i] = __ldcg(a.SX + size_t(i) * n + i) / __ldcg(a.G + size_t(i) * n + i);
      slf[i] = float(sl[i]);
    }
    __syncthreads();
    for (int c = tid; c < n; c += PR_THREADS) {
      const long long kc = pr_key(sl[c]);
      int r = 0;
      for (int o = 0; o < n; ++o) {
        const long long ko = pr_key(sl[o]);
        r += (ko > kc || (ko == kc && o < c)) ? 1 : 0;
      }
      rank[c] = r;
    }
    __syncthreads();
  };
  auto xtsx1 = [&]() {   // G = X^T X and B = F X or S X
    double tl;
    const double v = pr_products(g, n, X, X, n, a.G, true, a.F ? a.F : a.S, X, a.F ? a.m : n, a.B, n, tl, sA, sB);
    pr_block_pair(v, 0.0, red, a.part + g.b, nullptr);
  };
  auto xtsx2 = [&]() {                  // SX = B^T B or X^T B
    double tl;
    const double v = pr_products(g, n, a.F ? a.B : X, a.B, a.F ? a.m : n, a.SX, false, nullptr, nullptr, 0, nullptr, t0, tl,
                                 sA, sB);
    pr_block_pair(v, tl, red, a.part + G + g.b, a.part + 2 * G + g.b);
  };
  do {
    // ---- the level's start: X = Y, or X = V diag(I, Y)
    const int nt0 = n - t0;
    if (a.level == 0) {
      double f = 0.0;
      for (int e = g.b * PR_THREADS + tid; e < n * n; e += G * PR_THREADS) {
        X[e] = a.Y[e];
        f = fma(a.S[e], a.S[e], f);
      }
      f += __shfl_xor_sync(0xffffffffu, f, 1);
      f += __shfl_xor_sync(0xffffffffu, f, 2);
      pr_block_pair(f, 0.0, red, a.part + 3 * G + g.b, nullptr);
    } else {
      for (int e = g.b * PR_THREADS + tid; e < n * t0; e += G * PR_THREADS) {
        const int i = e / t0, j = e % t0;
        X[size_t(i) * n + j] = a.V[size_t(i) * n + j];
      }
      const int rt = (n + PR_T - 1) / PR_T, ct = (nt0 + PR_T - 1) / PR_T;
      const int l = tid & 3, oi = (tid >> 2) >> 3, oj = (tid >> 2) & 7;
      for (int t = g.b; t < rt * ct; t += G) {
        const int i0 = (t / ct) * PR_T, j0 = (t % ct) * PR_T;
        const double s = pr_tile(a.V + t0, n, false, i0, n, a.Y, nt0, j0, nt0, nt0, sA, sB);
        if (l == 0 && i0 + oi < n && j0 + oj < nt0) X[size_t(i0 + oi) * n + t0 + j0 + oj] = s;
      }
    }
    if (!(ok = pr_sync(st, g, target, &flag))) break;
    // ---- Newton-Schulz
    pr_products(g, n, X, X, n, a.G, true, nullptr, nullptr, 0, nullptr, n, unused, sA, sB);
    if (!(ok = pr_sync(st, g, target, &flag))) break;
    pr_update(g, n, X, a.G, Xn, 1, nullptr, sA, sB);
    swap();
    if (!(ok = pr_sync(st, g, target, &flag))) break;
    // ---- Ogita-Aishima iterations
    float before = 1.f;
    for (int it = 0; it < PR_MAX_IT; ++it) {
      xtsx1();
      if (!(ok = pr_sync(st, g, target, &flag))) break;
      xtsx2();
      if (!(ok = pr_sync(st, g, target, &flag))) break;
      // the resolution of the eigenvalue estimates, on the warps that lambda() leaves idle (n <= 128): one a
      // sum, then 2 (||off-diagonal|| + ||S|| ||X^T X - I||) and the same for the level's block
      if (tid >= 128) {
        const int q = (tid >> 5) - 4, lane = tid & 31;
        if (q < 3 || (a.level == 0 && it == 0)) {
          double v = 0.0;
          for (int i = lane; i < G; i += 32) v += __ldcg(a.part + q * G + i);
          for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (lane == 0) norms[q] = sqrt(v);
        } else if (it == 0 && lane == 0) {
          norms[3] = __ldcg(&st->anorm);
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (tid == 128) {
          delta_s = 2.0 * fma(norms[3], norms[0], norms[1]);
          // pairs with the level's block: with a factor their entries carry errors on their own
          // scale, so the couplings among the columns above it do not hold them back; the block's
          // largest eigenvalue comes from the level before
          delta_t = a.F ? 2.0 * fma(a.level > 0 && t0 < n ? __ldcg(a.lam + t0) : norms[3], norms[0], norms[2]) : delta_s;
        }
      }
      lambda();
      const double delta_all = delta_s, delta_tail = delta_t;
      // the next level's threshold, if its tail starts among the kept ones (it is then taken)
      // (comparisons in FP32: an FP64 one takes a slot of the FP64 pipe)
      const float fi_ = tid < n ? slf[tid] : 0.f;
      if (tid < n && rank[tid] == 0) tail_s = float(a.tau_next) * fi_;
      __syncthreads();
      const int below = __syncthreads_count(tid < n && fi_ < tail_s);
      const float tail = (tail_s > 0.f && below >= 2 && n - below < a.keep) ? tail_s : 0.f;
      float big = 0.f;
      for (int e = g.b * PR_THREADS + tid; e < n * n; e += G * PR_THREADS) {
        const int i = e / n, j = e % n;
        const double r = (i == j ? 1.0 : 0.0) - __ldcg(a.G + e);
        double v = 0.5 * r;
        // pairs that decide: across the cut, or across the next level's threshold and apart; of pairs
        // below that threshold the next level takes care
        const bool cut = (rank[i] < a.keep) != (rank[j] < a.keep);
        const float hi = fmaxf(slf[i], slf[j]), lo = fminf(slf[i], slf[j]);
        const bool across = cut || (tail > 0.f && hi >= tail && lo < tail && lo < 0.1f * hi);
        const bool decides = across && hi >= tail && max(i, j) >= t0;
        if (i != j) {
          // the kept space is what counts: a pair on one side of the cut takes small steps only
          // (a near-degenerate pair's first-order step of size t leaves X^T X - I at t^2, and its
          // two vectors span the same space as they are)
          const double d = sl[j] - sl[i];
          const double t = fma(sl[j], r, __ldcg(a.SX + e)) / d;
          if (fabs(d) > (max(i, j) < t0 ? delta_all : delta_tail) && (across || fabs(t) < PR_STEP)) v = t;
          if (decides) big = fmaxf(big, fminf(fabsf(float(t)), 1.f));   // also while it is not resolved
        }
        a.E[e] = v;
        if (a.keep == n) big = fmaxf(big, fabsf(float(v)));
      }
      for (int o = 16; o > 0; o >>= 1) big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, o));
      __syncthreads();
      if ((tid & 31) == 0) redf[tid >> 5] = big;
      __syncthreads();
      if (tid == 0) {
        for (int w = 1; w < PR_THREADS / 32; ++w) big = fmaxf(big, redf[w]);
        a.big[g.b] = big;
      }
      if (!(ok = pr_sync(st, g, target, &flag))) break;
      pr_update(g, n, X, a.E, Xn, 0, nullptr, sA, sB);
      swap();
      // the same decision in every CTA: the largest correction of this iteration
      float mb = 0.f;
      for (int i = tid & 31; i < G; i += 32) mb = fmaxf(mb, __ldcg(a.big + i));
      for (int o = 16; o > 0; o >>= 1) mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, o));
      if (!(ok = pr_sync(st, g, target, &flag))) break;
      // corrections shrink quadratically where the gaps resolve a pair, by a constant factor while a
      // cluster next to it is unresolved: mb^2 / before bounds the next one either way; a level at
      // its rounding floor no longer shrinks
      if (mb * (it ? mb / before : 1.f) < PR_STOP || (it >= 2 && mb > 0.3f * before && mb < float(PR_STEP))) break;
      before = mb;
    }
    if (!ok) break;
    // ---- Newton-Schulz, eigenvalues, and a last Newton-Schulz step into the sorted V
    pr_products(g, n, X, X, n, a.G, true, nullptr, nullptr, 0, nullptr, n, unused, sA, sB);
    if (!(ok = pr_sync(st, g, target, &flag))) break;
    pr_update(g, n, X, a.G, Xn, 1, nullptr, sA, sB);
    swap();
    if (!(ok = pr_sync(st, g, target, &flag))) break;
    xtsx1();
    if (!(ok = pr_sync(st, g, target, &flag))) break;
    xtsx2();
    if (!(ok = pr_sync(st, g, target, &flag))) break;
    lambda();
    pr_update(g, n, X, a.G, a.V, 1, rank, sA, sB);
    if (a.tau_next > 0.0)
      for (int e = g.b * PR_THREADS + tid; e < n * n; e += G * PR_THREADS)
        a.SXs[size_t(rank[e / n]) * n + rank[e % n]] = __ldcg(a.SX + e);
    if (g.b == 0) {
      if (a.level == 0 && tid == 0) st->anorm = norms[3];
      for (int i = tid; i < n; i += PR_THREADS) {
        a.lam[rank[i]] = sl[i];
        a.w[rank[i]] = ldexp(sl[i], st->e);
      }
    }
  } while (false);
  return ok;
}

// A level whose waits ran out is done again by the last CTA to leave it, alone and without waits, so that the
// results do not depend on the wait limit (slow: one SM's FP64 units; not needed while the grid is resident).
__global__ void __launch_bounds__(PR_THREADS, 2) k_psd_refine(PsdArgs a) {
  __shared__ unsigned int before;
  if (a.level > 0 && a.st->need == 0) return;
  PsdGrid g = {int(gridDim.x), int(blockIdx.x)};
  while (!psd_level(a, g)) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) before = atomicAdd(&a.st->left, 1u);
    __syncthreads();
    if (before != gridDim.x - 1) return;
    __threadfence();
    g = {1, 0};
  }
}

// The next level's tail block from the sorted eigenvalues: it holds the eigenvalues below tau
// times the largest, and is taken when there are at least two and it starts among the kept ones.
__global__ void k_psd_tail(int n, int keep, double tau, const double* __restrict__ lam, PsdState* st, int level) {
  if (level > 0 && st->need == 0) return;   // a level that was not taken ends the sequence
  const double top = lam[0];
  int c = 0;
  for (int i = threadIdx.x; i < n; i += 32) c += (top > 0.0 && lam[i] < tau * top) ? 1 : 0;
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (threadIdx.x == 0) {
    st->t0 = n - c;
    st->need = (c >= 2 && n - c < keep) ? 1 : 0;
  }
}

__global__ void k_psd_scale_factor(int64_t n, const double* __restrict__ F, double* __restrict__ Fc,
                                   const PsdState* __restrict__ st) {
  const int h = st->e / 2;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    Fc[i] = ldexp(F[i], -h);
}

size_t pr_smem(int n, int m) {
  const int K = std::max(n, m);
  return size_t(PR_T) * (2 * K + 2) * sizeof(double) + n * sizeof(double) + n * sizeof(int);
}

int g_psd_per_sm = -1;

}  // namespace

void eigh_psd_init_attributes() {
  if (g_psd_per_sm >= 0) return;
  QTT_CUDA(cudaFuncSetAttribute(k_psd_start, cudaFuncAttributeMaxDynamicSharedMemorySize, int(ps_smem(PS_MAX_N))));
  QTT_CUDA(cudaFuncSetAttribute(k_psd_refine, cudaFuncAttributeMaxDynamicSharedMemorySize, int(pr_smem(PS_MAX_N, 256))));
  int per_sm = 0;
  QTT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_psd_refine, PR_THREADS, pr_smem(PS_MAX_N, 256)));
  g_psd_per_sm = per_sm;
}

// Orders 2 to 128, where the start's matrix fits a CTA's shared memory.  Against the general solver, when this one came
// in (everything else the same): a sketched product at 20 bits (bond 64) 49.5 -> 23.5 ms, the encoding of 2^20 values
// 12.7 -> 3.2 ms; with the present QR 19.9 and 2.9 ms.  Rank 5 of 32 kept at order 64: 2.99 -> 0.46 ms.  Error against the
// exact decomposition of the same product 4e-13 .. 3e-11 -> 2e-13 (12 inputs).
bool eigh_psd_fits(int n, int m) {
  eigh_psd_init_attributes();
  return n >= 2 && n <= PS_MAX_N && m <= 256 && g_psd_per_sm >= 2;
}

void eigh_psd(Ctx& c, int n, const double* S, double* w, double* V, int keep, const double* F, int m) {
  if (keep <= 0 || keep > n) keep = n;
  const size_t nn = size_t(n) * n;
  const int nt = (n + PR_T - 1) / PR_T;
  // as many CTAs as the widest phase has tiles; one per SM on the caller's own stream, half of
  // that on worker streams (four products may run side by side; two CTAs fit an SM)
  const int tiles = nt * (nt + 1) / 2 + nt * (F ? (m + PR_T - 1) / PR_T : nt);
  const int G = std::max(1, std::min(tiles, &c == c.root ? c.num_sms : std::max(1, c.num_sms / 2)));
  DBuf Ssc(&c, nn), Y(&c, nn), X0(&c, nn), X1(&c, nn), Gm(&c, nn), B(&c, size_t(std::max(m, n)) * n), SX(&c, nn),
      E(&c, nn), SXs(&c, nn), lam(&c, size_t(n)), part(&c, size_t(5) * G), stb(&c, (sizeof(PsdState) + 7) / 8),
      Fsc(&c, F ? size_t(m) * n : 1);
  PsdState* st = reinterpret_cast<PsdState*>(stb.p);
  ProfScope ps(c, KC_EIG);
  k_psd_start<<<1, PS_THREADS, ps_smem(n), c.stream>>>(n, S, F ? 1 : 0, Ssc.p, Y.p, st, 0, c.root->wait_ns);
  after_launch(c, "psd_start");
  if (F) {
    k_psd_scale_factor<<<unsigned(std::min<int64_t>((int64_t(m) * n + 255) / 256, 1024)), 256, 0, c.stream>>>(
        int64_t(m) * n, F, Fsc.p, st);
    after_launch(c, "psd_scale_factor");
  }
  const double taus[4] = {1e-8, 1e-16, 1e-24, 0.0};
  const int levels = F ? 4 : 2;
  PsdArgs a;
  a.n = n; a.m = F ? m : 0; a.keep = keep;
  a.S = Ssc.p; a.F = F ? Fsc.p : nullptr; a.Y = Y.p; a.V = V; a.w = w; a.lam = lam.p;
  a.X0 = X0.p; a.X1 = X1.p; a.G = Gm.p; a.B = B.p; a.SX = SX.p; a.E = E.p; a.SXs = SXs.p;
  a.part = part.p;
  a.big = reinterpret_cast<float*>(part.p + 4 * size_t(G));
  a.st = st;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(G));
  cfg.blockDim = dim3(PR_THREADS);
  cfg.dynamicSmemBytes = pr_smem(n, a.m);
  cfg.stream = c.stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  for (int level = 0; level < levels; ++level) {
    a.level = level;
    const bool last = level == levels - 1;
    a.tau_next = last ? 0.0 : taus[level];
    if (level > 0) {
      k_psd_start<<<1, PS_THREADS, ps_smem(n), c.stream>>>(n, SXs.p, 0, nullptr, Y.p, st, level, c.root->wait_ns);
      after_launch(c, "psd_start");
    }
    QTT_CUDA(cudaLaunchKernelEx(&cfg, k_psd_refine, a));
    after_launch(c, "psd_refine");
    if (!last) {
      k_psd_tail<<<1, 32, 0, c.stream>>>(n, keep, taus[level], lam.p, st, level);
      after_launch(c, "psd_tail");
    }
  }
}

}  // namespace qtt

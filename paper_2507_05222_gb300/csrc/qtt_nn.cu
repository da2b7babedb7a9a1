// Learned warm start of the Poisson solve: a small convolutional network on a coarse (eta, xi)
// grid, trained on states the solver itself produces, predicting the pressure change of the
// next step (the growth direction standing in for the paper's unspecified preconditioner of
// the Poisson sweeps, Sec. IV.C / App. G).  Hand-written FP32 kernels: 3 x 3 convolution
// forward, its data and weight gradients, ReLU mask, squared-error loss, Adam (Kingma & Ba
// 2015), and the coarse/fine grid transfers.
//
// Convolution: y[n, o, i, j] = b[o] + sum_{c, a, e} w[o, c, a, e] x[n, c, i + a - 1, j + e - 1],
// zero outside the eta range (first axis: the wall and the far field are not neighbours),
// periodic in xi (second axis, angular).  Layout NCHW; parameters one flat vector, layer by
// layer: weights (c_out, c_in, 3, 3) then bias (c_out).
#include <algorithm>
#include <cmath>
#include <vector>

#include "qtt_internal.h"
#include "qtt_nn.h"

namespace qtt {

namespace {

constexpr float NN_B1 = 0.9f, NN_B2 = 0.999f, NN_EPS = 1e-8f;

unsigned nn_blocks(int64_t n, int t) { return unsigned(std::min<int64_t>((n + t - 1) / t, 65535 * 8)); }

// The convolution and its data gradient, for large layers.  FLIP = false: out[n, o] = b[o] + sum_c w[o, c] * in[n, c]
// (with ReLU, and the layer's input affine (x - shift[c]) scale[c], zero outside the grid in the
// mapped values); FLIP = true: out[n, c] = sum_o w[o, c] (transposed stencil) in[n, o], zero where
// the activation `act` of the layer below is not positive (its ReLU).  A CTA computes an R x 32
// tile of pixels for 4 COT channels: a thread has four neighbouring pixels of COT channels in
// registers, input rows and weights staged in shared memory CC input channels at a time, so that
// 36 COT multiply-adds take 18 + 9 COT / 4 shared loads, where one thread
// per output (k_conv_direct) loads an input and a weight for each multiply-add.  The order of each output's sum is
// unchanged (input channels, then taps).  What bounds it is the latency of a stage's loads between its two barriers:
// the FMA pipe is 33 to 40 % busy, the issue slots 58 to 60 %, at 2.5 warps a scheduler.  With k_conv_wgrad a training step
// of 8 x 128 x 128 cells, width 32, depth 4 (15 GFLOP) went from 14.4 to 0.97 ms.
template <bool FLIP>
__global__ void __launch_bounds__(256) k_conv(int ni, int no, int H, int W, const float* __restrict__ in,
                                              const float* __restrict__ shift, const float* __restrict__ scale,
                                              const float* __restrict__ w, const float* __restrict__ b,
                                              const float* __restrict__ act, float* __restrict__ out, int relu) {
  constexpr int COT = 8;                         // output channels of a thread
  constexpr int CC = 4;                          // input channels per stage
  constexpr int NG = 4;                          // channel groups of a CTA
  constexpr int R = 256 / NG / 8;                // tile rows (8 threads of four pixels a row)
  constexpr int CO = COT * NG;
  __shared__ float xs[CC][R + 2][36];
  __shared__ __align__(16) float ws[CC][9][CO];
  const int tid = threadIdx.x;
  const int px = tid & 7, py = (tid >> 3) % R, og = tid / (8 * R);
  const int tw = (W + 31) / 32, th = (H + R - 1) / R;
  const int n = blockIdx.x / (tw * th), t = blockIdx.x % (tw * th);
  const int i0 = (t / tw) * R, j0 = (t % tw) * 32, o0 = blockIdx.y * CO;
  const int64_t per = int64_t(H) * W;
  // rows of the stencil that lie outside the grid are left out, not multiplied by zero: a weight that is
  // not finite has no effect there (fmaxf would turn its NaN into a plausible 0)
  const bool up = i0 + py > 0, down = i0 + py + 1 < H;
  float acc[COT][4];
#pragma unroll
  for (int o = 0; o < COT; ++o) {
    const int oo = o0 + og * COT + o;
    const float bv = (!FLIP && oo < no) ? b[oo] : 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[o][q] = bv;
  }
  for (int c0 = 0; c0 < ni; c0 += CC) {
    __syncthreads();
    for (int e = tid; e < CC * (R + 2) * 34; e += 256) {
      const int c = e / ((R + 2) * 34), r = (e / 34) % (R + 2), q = e % 34;
      const int ii = i0 + r - 1, ch = c0 + c;
      int jj = j0 + q - 1;
      jj = jj < 0 ? jj + W : jj;
      while (jj >= W) jj -= W;                   // periodic; columns beyond the grid are not written out
      float v = 0.f;
      if (ch < ni && ii >= 0 && ii < H) {
        v = in[(int64_t(n) * ni + ch) * per + int64_t(ii) * W + jj];
        if (!FLIP && shift) v = (v - shift[ch]) * scale[ch];
      }
      xs[c][r][q] = v;
    }
    for (int e = tid; e < CC * 9 * CO; e += 256) {
      const int c = e / (9 * CO), k = (e / CO) % 9, o = e % CO;
      const int ch = c0 + c, oo = o0 + o;
      float v = 0.f;
      if (ch < ni && oo < no) v = FLIP ? w[(int64_t(ch) * no + oo) * 9 + k] : w[(int64_t(oo) * ni + ch) * 9 + k];
      ws[c][k][o] = v;
    }
    __syncthreads();
    const int nc = min(CC, ni - c0);
    for (int c = 0; c < nc; ++c) {
      float x[3][6];
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int q = 0; q < 6; ++q) x[a][q] = xs[c][py + a][4 * px + q];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int ra = FLIP ? 2 - a : a;
        if ((ra == 0 && !up) || (ra == 2 && !down)) continue;
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          const int re = FLIP ? 2 - e : e;
#pragma unroll
          for (int o = 0; o < COT; o += 4) {
            const float4 wv = *reinterpret_cast<const float4*>(&ws[c][a * 3 + e][og * COT + o]);
            const float wq[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
              for (int q = 0; q < 4; ++q) acc[o + u][q] = fmaf(wq[u], x[ra][q + re], acc[o + u][q]);
          }
        }
      }
    }
  }
  const int i = i0 + py;
  if (i >= H) return;
#pragma unroll
  for (int o = 0; o < COT; ++o) {
    const int oo = o0 + og * COT + o;
    if (oo >= no) continue;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = j0 + 4 * px + q;
      if (j >= W) continue;
      const int64_t g = (int64_t(n) * no + oo) * per + int64_t(i) * W + j;
      float v = acc[o][q];
      if (FLIP) v = act[g] > 0.f ? v : 0.f;
      else if (relu) v = fmaxf(v, 0.f);
      out[g] = v;
    }
  }
}

// The same with one thread per output, for small layers: a load for each multiply-add, but no stages, so
// the time is that of one output's chain until the grid fills the chip.
template <bool FLIP>
__global__ void __launch_bounds__(256) k_conv_direct(int B, int ni, int no, int H, int W, const float* __restrict__ in,
                                                     const float* __restrict__ shift, const float* __restrict__ scale,
                                                     const float* __restrict__ w, const float* __restrict__ b,
                                                     const float* __restrict__ act, float* __restrict__ out, int relu) {
  const int64_t total = int64_t(B) * no * H * W, per = int64_t(H) * W;
  for (int64_t idx = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; idx < total; idx += int64_t(gridDim.x) * blockDim.x) {
    const int64_t plane = idx / per;
    const int at = int(idx - plane * per), i = at / W, j = at - i * W;
    const int n = int(plane / no), o = int(plane - int64_t(n) * no);
    int jc[3];
    jc[0] = j == 0 ? W - 1 : j - 1;
    jc[1] = j;
    jc[2] = j == W - 1 ? 0 : j + 1;
    float s = FLIP ? 0.f : b[o];
    for (int c = 0; c < ni; ++c) {
      const float* xc = in + (int64_t(n) * ni + c) * per;
      const float* wc = FLIP ? w + (int64_t(c) * no + o) * 9 : w + (int64_t(o) * ni + c) * 9;
      const bool affine = !FLIP && shift;
      const float sh = affine ? shift[c] : 0.f, sc = affine ? scale[c] : 1.f;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int ii = FLIP ? i - a + 1 : i + a - 1;
        const bool inside = ii >= 0 && ii < H;
        const float* row = xc + int64_t(inside ? ii : i) * W;
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          float v = row[jc[FLIP ? 2 - e : e]];
          if (affine) v = (v - sh) * sc;
          s = inside ? fmaf(wc[a * 3 + e], v, s) : s;
        }
      }
    }
    if (FLIP) s = act[idx] > 0.f ? s : 0.f;
    else if (relu) s = fmaxf(s, 0.f);
    out[idx] = s;
  }
}

// Weight and bias gradients of a small layer, one CTA per value: [0, co ci 9) the weights (o, c, a, e), then
// the biases, written in that order.  Fixed summation order.
__global__ void __launch_bounds__(256) k_conv_wgrad_direct(int B, int ci, int co, int H, int W, const float* __restrict__ x,
                                                           const float* __restrict__ shift, const float* __restrict__ scale,
                                                           const float* __restrict__ dy, float* __restrict__ grad) {
  __shared__ float red[8];
  const int nw = co * ci * 9, blk = blockIdx.x;
  const bool bias = blk >= nw;
  const int o = bias ? blk - nw : blk / (ci * 9), k = bias ? 0 : blk % (ci * 9), c = k / 9, a = (k % 9) / 3, e = k % 3;
  const float sh = !bias && shift ? shift[c] : 0.f, sc = !bias && shift ? scale[c] : 1.f;
  const int per = H * W, total = B * per;
  float s = 0.f;
  for (int t = threadIdx.x; t < total; t += 256) {
    const int n = t / per, at = t - n * per, i = at / W, j = at - i * W;
    const float g = dy[(int64_t(n) * co + o) * per + at];
    const int ii = i + a - 1;
    int jj = j + e - 1;
    jj = jj < 0 ? jj + W : jj >= W ? jj - W : jj;
    if (bias) s += g;
    else if (ii >= 0 && ii < H) s = fmaf(g, (x[(int64_t(n) * ci + c) * per + int64_t(ii) * W + jj] - sh) * sc, s);
  }
  for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = red[threadIdx.x & 7];
    for (int q = 4; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
    if (threadIdx.x == 0) grad[blk] = s;
  }
}

constexpr int CW_TR = 4, CW_TC = 32, CW_CH = 32, CW_XS = 34, CW_YS = 36;   // k_conv_wgrad

// One row of a tile: xr the input row above it, yr the row of dy; with TEST, the input rows above and below only where
// they are in the grid (up, down).
template <bool TEST>
__device__ __forceinline__ void cw_row(const float* xr, const float* yr, bool bias, bool up, bool down, float (&acc)[4][2][9],
                                       float (&bs)[4]) {
  float2 win[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int e = 0; e < 2; ++e) win[a][e + 1] = *reinterpret_cast<const float2*>(xr + (a * (CW_TC + 2) + e) * CW_XS);
#pragma unroll (TEST ? 1 : 4)
  for (int q = 0; q < CW_TC; ++q) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      win[a][0] = win[a][1];
      win[a][1] = win[a][2];
      win[a][2] = *reinterpret_cast<const float2*>(xr + (a * (CW_TC + 2) + q + 2) * CW_XS);
    }
    const float4 g4 = *reinterpret_cast<const float4*>(yr + q * CW_YS);
    const float g[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      if (bias) bs[o] += g[o];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        if (TEST && ((a == 0 && !up) || (a == 2 && !down))) continue;
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          acc[o][0][3 * a + e] = fmaf(g[o], win[a][e].x, acc[o][0][3 * a + e]);
          acc[o][1][3 * a + e] = fmaf(g[o], win[a][e].y, acc[o][1][3 * a + e]);
        }
      }
    }
  }
}

// Weight and bias gradients: part[g][(o ci + c) 9 + tap] and part[g][co ci 9 + o] = the sums over the
// pixel tiles g, g + gridDim.x, ... of dy[n, o, i, j] x'[n, c, i + a - 1, j + e - 1] (x' with the
// layer's input affine) and of dy.  A CTA keeps a chunk of 32 x 32 channel pairs: a thread has the
// nine taps of 4 x 2 of them (72 sums) in registers and slides a 3 x 3 window along the rows of a
// 4 x 32 tile staged in shared memory; where the layer has fewer channels the threads share the
// tile's rows instead (pg).  The partial sums are added by k_conv_wsum in a fixed order.  (One CTA
// per weight reads both activations from L2 for every one of the 9 co ci weights.)
__global__ void __launch_bounds__(256, 2) k_conv_wgrad(int B, int ci, int co, int H, int W, const float* __restrict__ x,
                                                    const float* __restrict__ shift, const float* __restrict__ scale,
                                                    const float* __restrict__ dy, float* __restrict__ part) {
  extern __shared__ __align__(16) float cw_sm[];
  float* xs = cw_sm;                                          // [(TR + 2)][TC + 2][CW_XS]
  float* ys = xs + (CW_TR + 2) * (CW_TC + 2) * CW_XS;         // [TR][TC][CW_YS]
  const int tid = threadIdx.x;
  const int o0 = (blockIdx.y % ((co + CW_CH - 1) / CW_CH)) * CW_CH, c0 = (blockIdx.y / ((co + CW_CH - 1) / CW_CH)) * CW_CH;
  const int no = min(CW_CH, co - o0), nc = min(CW_CH, ci - c0);
  const int OG = (no + 3) / 4, CG = (nc + 1) / 2, PG = min(CW_TR, 256 / (OG * CG));
  const int og = tid % OG, cg = (tid / OG) % CG, pg = tid / (OG * CG);
  const int64_t per = int64_t(H) * W;
  const int tw = (W + CW_TC - 1) / CW_TC, th = (H + CW_TR - 1) / CW_TR, ntiles = B * tw * th;
  float acc[4][2][9], bs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int o = 0; o < 4; ++o)
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int k = 0; k < 9; ++k) acc[o][c][k] = 0.f;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int n = t / (tw * th), i0 = ((t / tw) % th) * CW_TR, j0 = (t % tw) * CW_TC;
    __syncthreads();
    int top = 0;                                              // largest magnitude staged, as an integer
    for (int e = tid; e < CW_CH * (CW_TR + 2) * (CW_TC + 2); e += 256) {
      const int q = e % (CW_TC + 2), r = (e / (CW_TC + 2)) % (CW_TR + 2), c = e / ((CW_TC + 2) * (CW_TR + 2));
      const int ii = i0 + r - 1;
      int jj = j0 + q - 1;
      jj = jj < 0 ? jj + W : jj;
      while (jj >= W) jj -= W;
      float v = 0.f;
      if (c < nc && ii >= 0 && ii < H) {
        v = x[(int64_t(n) * ci + c0 + c) * per + int64_t(ii) * W + jj];
        if (shift) v = (v - shift[c0 + c]) * scale[c0 + c];
      }
      xs[(r * (CW_TC + 2) + q) * CW_XS + c] = v;
      top = max(top, __float_as_int(v) & 0x7fffffff);
    }
    for (int e = tid; e < CW_CH * CW_TR * CW_TC; e += 256) {
      const int q = e % CW_TC, r = (e / CW_TC) % CW_TR, o = e / (CW_TC * CW_TR);
      const int ii = i0 + r, jj = j0 + q;
      const float v = (o < no && ii < H && jj < W) ? dy[(int64_t(n) * co + o0 + o) * per + int64_t(ii) * W + jj] : 0.f;
      ys[(r * CW_TC + q) * CW_YS + o] = v;
      top = max(top, __float_as_int(v) & 0x7fffffff);
    }
    // Rows outside the grid count as zeros, which a value that is not finite must not meet (they are no part of the
    // sums): a tile with such a value takes its rows with the test, which in every tile cost 9 us of a 104 us step.
    const bool finite = __syncthreads_or(top >= 0x7f800000) == 0;
    if (pg < PG) {
      for (int r = pg; r < (finite ? CW_TR : min(CW_TR, H - i0)); r += PG) {
        const float* xr = xs + r * (CW_TC + 2) * CW_XS + 2 * cg;
        const float* yr = ys + r * CW_TC * CW_YS + 4 * og;
        if (finite) cw_row<false>(xr, yr, cg == 0, true, true, acc, bs);
        else cw_row<true>(xr, yr, cg == 0, i0 + r > 0, i0 + r + 1 < H, acc, bs);
      }
    }
  }
  // the row groups' sums, in order, into shared memory, then out
  __syncthreads();
  float* red = cw_sm;                                          // [32][32][9] then [32]
  for (int p = 0; p < PG; ++p) {
    if (pg == p) {
#pragma unroll
      for (int o = 0; o < 4; ++o) {
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int k = 0; k < 9; ++k) {
            float* d = &red[((4 * og + o) * CW_CH + 2 * cg + c) * 9 + k];
            *d = p == 0 ? acc[o][c][k] : *d + acc[o][c][k];
          }
        if (cg == 0) {
          float* d = &red[CW_CH * CW_CH * 9 + 4 * og + o];
          *d = p == 0 ? bs[o] : *d + bs[o];
        }
      }
    }
    __syncthreads();
  }
  float* dst = part + int64_t(blockIdx.x) * (int64_t(co) * ci * 9 + co);
  for (int e = tid; e < no * nc * 9; e += 256) {
    const int o = e / (nc * 9), c = (e / 9) % nc, k = e % 9;
    dst[(int64_t(o0 + o) * ci + c0 + c) * 9 + k] = red[(o * CW_CH + c) * 9 + k];
  }
  if (c0 == 0)
    for (int o = tid; o < no; o += 256) dst[int64_t(co) * ci * 9 + o0 + o] = red[CW_CH * CW_CH * 9 + o];
}
constexpr size_t kWgradSmem = ((CW_TR + 2) * (CW_TC + 2) * CW_XS + CW_TR * CW_TC * CW_YS) * sizeof(float);
static_assert(kWgradSmem >= (CW_CH * CW_CH * 9 + CW_CH) * sizeof(float), "wgrad reduction buffer");

// grad[e] = sum_g part[g][e], eight lanes a value, four sums a lane (strided over g), then a fixed tree: one
// chain of G / 8 additions a lane left gradients up to 24 % further from the 64-bit ones.
__global__ void __launch_bounds__(256) k_conv_wsum(int64_t n, int G, const float* __restrict__ part, float* __restrict__ grad) {
  const int64_t e = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 3;
  const int l = threadIdx.x & 7;
  float s4[4] = {0.f, 0.f, 0.f, 0.f};
  if (e < n) {
    int g = l;
#pragma unroll 2
    for (; g + 24 < G; g += 32)
#pragma unroll
      for (int q = 0; q < 4; ++q) s4[q] += part[int64_t(g + 8 * q) * n + e];
#pragma unroll
    for (int q = 0; q < 3; ++q)
      if (g + 8 * q < G) s4[q] += part[int64_t(g + 8 * q) * n + e];
  }
  float s = (s4[0] + s4[1]) + (s4[2] + s4[3]);
  for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (e < n && l == 0) grad[e] = s;
}

// dpred = 2 (pred - y / out_scale) / n and, per block, the sum of squared differences.
constexpr int MSE_BLOCKS = 256;
__global__ void __launch_bounds__(256) k_mse(int64_t n, const float* __restrict__ pred, const float* __restrict__ y,
                                             float inv_out, float* __restrict__ dpred, double* __restrict__ part) {
  __shared__ double red[8];
  double s = 0.0;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const float d = pred[i] - y[i] * inv_out;
    dpred[i] = 2.f * d / float(n);
    s += double(d) * d;
  }
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < 8; ++w) v += red[w];
    part[blockIdx.x] = v;
  }
}

// *loss = mean of the blocks' sums (fixed order)
__global__ void k_mse_sum(int64_t n, int G, const double* __restrict__ part, float* __restrict__ loss) {
  double v = 0.0;
  for (int i = threadIdx.x; i < G; i += 32) v += part[i];
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  if (threadIdx.x == 0) *loss = float(v / double(n));
}

__global__ void k_adam(int64_t n, float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, float lr, float bc1, float bc2) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const float gi = g[i];
    const float mi = NN_B1 * m[i] + (1.f - NN_B1) * gi;
    const float vi = NN_B2 * v[i] + (1.f - NN_B2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + NN_EPS);
  }
}

__global__ void k_scale(int64_t n, float* __restrict__ x, float s) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    x[i] *= s;
}

// coarse[I, J] = mean of the s x s block of fine (row-major (Hc s) x (Wc s)), s = 2^levels
__global__ void k_restrict(int Hc, int Wc, int s, const double* __restrict__ fine, float* __restrict__ coarse) {
  const int64_t total = int64_t(Hc) * Wc;
  for (int64_t idx = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; idx < total;
       idx += int64_t(gridDim.x) * blockDim.x) {
    const int I = int(idx / Wc), J = int(idx % Wc);
    const int64_t Wf = int64_t(Wc) * s;
    double acc = 0.0;
    for (int a = 0; a < s; ++a)
      for (int e = 0; e < s; ++e) acc += fine[(int64_t(I) * s + a) * Wf + int64_t(J) * s + e];
    coarse[idx] = float(acc / (double(s) * s));
  }
}

// one cell-centred bilinear doubling: (H x W) -> (2H x 2W), clamped in eta, periodic in xi
__global__ void k_prolong2(int H, int W, const double* __restrict__ c, double* __restrict__ f) {
  const int64_t total = int64_t(4) * H * W;
  for (int64_t idx = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; idx < total;
       idx += int64_t(gridDim.x) * blockDim.x) {
    const int i = int(idx / (2 * W)), j = int(idx % (2 * W));
    const int I = i >> 1, J = j >> 1;
    const int I2 = (i & 1) ? min(I + 1, H - 1) : max(I - 1, 0);
    const int J2 = (j & 1) ? (J + 1) % W : (J - 1 + W) % W;
    const double t1 = 0.75 * c[int64_t(I) * W + J] + 0.25 * c[int64_t(I2) * W + J];
    const double t2 = 0.75 * c[int64_t(I) * W + J2] + 0.25 * c[int64_t(I2) * W + J2];
    f[idx] = 0.75 * t1 + 0.25 * t2;
  }
}

__global__ void k_to_double(int64_t n, const float* __restrict__ x, double* __restrict__ y) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    y[i] = double(x[i]);
}

// mean and root mean square (one block, fixed order)
__global__ void k_moments(int64_t n, const float* __restrict__ x, double* __restrict__ out) {
  __shared__ double red[2][32];
  double s = 0.0, q = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
    const double v = x[i];
    s += v;
    q += v * v;
  }
  for (int off = 16; off > 0; off >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, off);
    q += __shfl_xor_sync(0xffffffffu, q, off);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = s;
    red[1][threadIdx.x >> 5] = q;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    double a = threadIdx.x < (blockDim.x >> 5) ? red[0][threadIdx.x] : 0.0;
    double b = threadIdx.x < (blockDim.x >> 5) ? red[1][threadIdx.x] : 0.0;
    for (int off = 16; off > 0; off >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, off);
      b += __shfl_xor_sync(0xffffffffu, b, off);
    }
    if (threadIdx.x == 0) {
      out[0] = a / double(n);
      out[1] = sqrt(b / double(n));
    }
  }
}

// Direct up to 2^19 outputs and for at most four output channels (the tiled kernel has 32), tiled above.  us
// a layer (mean over a network's), direct / tiled: 2 x 16 x 16 cells, width 32 13 / 31; 2 x 128 x 16, width 24
// 12 / 25; 8 x 64 x 48, width 32 42 / 26; 8 x 64 x 64 59 / 30; 8 x 128 x 128 205 / 76.  One output channel:
// 8 x 64 x 64 20 / 58.
constexpr int64_t kConvDirect = int64_t(1) << 19;     // outputs
// Direct up to 2^21 multiply-adds over at most 4096 pixels (16 a thread).  us a layer (mean over a network's),
// direct / tiled with its sum: 32 x 16 cells, width 12 4.2 / 14.6; 4 x 32 x 48, width 16 40 / 15; 8 x 128 x 128,
// width 32 3156 / 81.  A layer of one by 8 channels on 128 x 128 cells took 27 direct, its network's layers 11.5
// tiled.
constexpr int64_t kWgradDirect = int64_t(1) << 21, kWgradDirectPixels = 4096;
template <bool FLIP>
void conv(Ctx& c, int B, int ni, int no, int H, int W, const float* in, const float* shift, const float* scale,
          const float* w, const float* b, const float* act, float* out, int relu) {
  const int64_t outputs = int64_t(B) * no * H * W, tiles = int64_t(B) * ((W + 31) / 32) * ((H + 7) / 8);
  if (no <= 4 || outputs <= kConvDirect)
    k_conv_direct<FLIP><<<nn_blocks(outputs, 256), 256, 0, c.stream>>>(B, ni, no, H, W, in, shift, scale, w, b, act, out, relu);
  else
    k_conv<FLIP><<<dim3(unsigned(tiles), unsigned((no + 31) / 32)), 256, 0, c.stream>>>(ni, no, H, W, in, shift, scale, w, b,
                                                                                       act, out, relu);
  after_launch(c, FLIP ? "nn_conv_bwd_data" : "nn_conv_fwd");
}

float* fbuf(DBuf& b, Ctx& c, int64_t nfloats) {
  b.reset(&c, size_t((nfloats + 1) / 2));
  return reinterpret_cast<float*>(b.p);
}

}  // namespace

static void init_nn_attributes() {
  static bool done = false;
  if (done) return;
  QTT_CUDA(cudaFuncSetAttribute(k_conv_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kWgradSmem)));
  done = true;
}

int64_t nn_param_count(int c_in, int width, int depth) {
  int64_t n = 0;
  for (int k = 0; k < depth; ++k) {
    const int ci = k == 0 ? c_in : width, co = k == depth - 1 ? 1 : width;
    n += int64_t(co) * ci * 9 + co;
  }
  return n;
}

Net::Net(Ctx& c, int c_in_, int width_, int depth_, const float* params_host)
    : ctx(&c), c_in(c_in_), width(width_), depth(depth_) {
  QTT_CHECK_ARG(c_in >= 1 && c_in <= 64 && width >= 1 && width <= 256 && depth >= 1 && depth <= 16,
                "nn: 1 <= c_in <= 64, 1 <= width <= 256, 1 <= depth <= 16");
  nparam = nn_param_count(c_in, width, depth);
  for (int k = 0; k < depth; ++k) {
    const int ci = k == 0 ? c_in : width, co = k == depth - 1 ? 1 : width;
    ci_.push_back(ci);
    co_.push_back(co);
  }
  // one block of the context's pool: parameters, both moments, gradient, input affine
  const int64_t np = (nparam + 3) / 4 * 4;
  params = fbuf(store, c, 4 * np + 2 * c_in);
  m = params + np;
  v = m + np;
  grad = v + np;
  shift = grad + np;
  scale = shift + c_in;
  QTT_CUDA(cudaMemcpyAsync(params, params_host, size_t(nparam) * sizeof(float), cudaMemcpyHostToDevice, c.stream));
  QTT_CUDA(cudaMemsetAsync(m, 0, size_t(nparam) * sizeof(float), c.stream));
  QTT_CUDA(cudaMemsetAsync(v, 0, size_t(nparam) * sizeof(float), c.stream));
  std::vector<float> zero(c_in, 0.f), one(c_in, 1.f);
  QTT_CUDA(cudaMemcpyAsync(shift, zero.data(), size_t(c_in) * sizeof(float), cudaMemcpyHostToDevice, c.stream));
  QTT_CUDA(cudaMemcpyAsync(scale, one.data(), size_t(c_in) * sizeof(float), cudaMemcpyHostToDevice, c.stream));
  QTT_CUDA(cudaStreamSynchronize(c.stream));
}

Net::~Net() {
  if (ctx) cudaStreamSynchronize(ctx->stream);
}

void Net::set_scaling(const float* in_shift, const float* in_scale, float out_scale_) {
  QTT_CHECK_ARG(std::isfinite(out_scale_) && out_scale_ != 0.f, "nn: out_scale must be finite and non-zero");
  for (int c = 0; c < c_in; ++c)
    QTT_CHECK_ARG(std::isfinite(in_shift[c]) && std::isfinite(in_scale[c]), "nn: non-finite input scaling");
  QTT_CUDA(cudaMemcpyAsync(shift, in_shift, size_t(c_in) * sizeof(float), cudaMemcpyHostToDevice, ctx->stream));
  QTT_CUDA(cudaMemcpyAsync(scale, in_scale, size_t(c_in) * sizeof(float), cudaMemcpyHostToDevice, ctx->stream));
  QTT_CUDA(cudaStreamSynchronize(ctx->stream));
  out_scale = out_scale_;
}

// Forward pass over B samples of c_in x H x W; acts[k] = output of layer k (ReLU applied to
// all but the last).  Returns the last activation (B x H x W, in units of out_scale).
void Net::forward(int B, int H, int W, const float* x, std::vector<DBuf>& acts) {
  Ctx& c = *ctx;
  acts.resize(depth);
  int64_t off = 0;
  const float* in = x;
  for (int k = 0; k < depth; ++k) {
    const int ci = ci_[k], co = co_[k];
    float* out = fbuf(acts[k], c, int64_t(B) * co * H * W);
    const float* w = params + off;
    const float* b = w + int64_t(co) * ci * 9;
    conv<false>(c, B, ci, co, H, W, in, k == 0 ? shift : nullptr, k == 0 ? scale : nullptr, w, b, nullptr, out,
                k < depth - 1 ? 1 : 0);
    off += int64_t(co) * ci * 9 + co;
    in = out;
  }
}

void Net::predict(int B, int H, int W, const float* x, float* y) {
  std::vector<DBuf> acts;
  forward(B, H, W, x, acts);
  const int64_t n = int64_t(B) * H * W;
  QTT_CUDA(cudaMemcpyAsync(y, acts[depth - 1].p, size_t(n) * sizeof(float), cudaMemcpyDeviceToDevice, ctx->stream));
  if (out_scale != 1.f) {
    k_scale<<<nn_blocks(n, 256), 256, 0, ctx->stream>>>(n, y, out_scale);
    after_launch(*ctx, "nn_scale");
  }
}

float Net::train_step(int B, int H, int W, const float* x, const float* y, float lr, float* loss_dev) {
  Ctx& c = *ctx;
  std::vector<DBuf> acts;
  forward(B, H, W, x, acts);
  const int64_t per = int64_t(H) * W;
  DBuf dyb, dxb;
  float* dy = fbuf(dyb, c, int64_t(B) * per);
  DBuf mpart(&c, MSE_BLOCKS);
  const int mg = int(std::min<int64_t>(MSE_BLOCKS, (int64_t(B) * per + 255) / 256));
  k_mse<<<mg, 256, 0, c.stream>>>(int64_t(B) * per, reinterpret_cast<float*>(acts[depth - 1].p), y, 1.f / out_scale, dy,
                                  mpart.p);
  after_launch(c, "nn_mse");
  k_mse_sum<<<1, 32, 0, c.stream>>>(int64_t(B) * per, mg, mpart.p, loss_dev);
  after_launch(c, "nn_mse_sum");
  init_nn_attributes();
  // parameter offsets per layer
  std::vector<int64_t> offs(depth);
  int64_t off = 0;
  for (int k = 0; k < depth; ++k) {
    offs[k] = off;
    off += int64_t(co_[k]) * ci_[k] * 9 + co_[k];
  }
  for (int k = depth - 1; k >= 0; --k) {
    const int ci = ci_[k], co = co_[k];
    const float* in = k == 0 ? x : reinterpret_cast<float*>(acts[k - 1].p);
    float* dw = grad + offs[k];
    const int64_t nw = int64_t(co) * ci * 9 + co;
    if (B * per <= kWgradDirectPixels && (nw - co) * B * per <= kWgradDirect) {
      k_conv_wgrad_direct<<<unsigned(nw), 256, 0, c.stream>>>(B, ci, co, H, W, in, k == 0 ? shift : nullptr,
                                                              k == 0 ? scale : nullptr, dy, dw);
      after_launch(c, "nn_conv_wgrad");
    } else {
      const int64_t tiles = int64_t(B) * ((W + CW_TC - 1) / CW_TC) * ((H + CW_TR - 1) / CW_TR);
      const int chunks = ((co + CW_CH - 1) / CW_CH) * ((ci + CW_CH - 1) / CW_CH);
      const int G = int(std::min<int64_t>(tiles, std::max(1, 2 * c.num_sms / chunks)));   // two CTAs per SM
      DBuf wpart;
      float* wp = fbuf(wpart, c, nw * G);
      k_conv_wgrad<<<dim3(unsigned(G), unsigned(chunks)), 256, kWgradSmem, c.stream>>>(
          B, ci, co, H, W, in, k == 0 ? shift : nullptr, k == 0 ? scale : nullptr, dy, wp);
      after_launch(c, "nn_conv_wgrad");
      k_conv_wsum<<<unsigned((nw * 8 + 255) / 256), 256, 0, c.stream>>>(nw, G, wp, dw);
      after_launch(c, "nn_conv_wsum");
    }
    if (k > 0) {
      float* dx = fbuf(dxb, c, int64_t(B) * ci * per);
      conv<true>(c, B, co, ci, H, W, dy, nullptr, nullptr, params + offs[k], nullptr,
                 reinterpret_cast<float*>(acts[k - 1].p), dx, 0);
      std::swap(dyb, dxb);
      dy = reinterpret_cast<float*>(dyb.p);
    }
  }
  ++t;
  const float bc1 = 1.f - std::pow(NN_B1, float(t)), bc2 = 1.f - std::pow(NN_B2, float(t));
  k_adam<<<nn_blocks(nparam, 256), 256, 0, c.stream>>>(nparam, params, grad, m, v, lr, bc1, bc2);
  after_launch(c, "nn_adam");
  float h = 0.f;
  QTT_CUDA(cudaMemcpyAsync(&h, loss_dev, sizeof(float), cudaMemcpyDeviceToHost, c.stream));
  QTT_CUDA(cudaStreamSynchronize(c.stream));
  return h;
}

void grid_restrict(Ctx& c, int Hc, int Wc, int levels, const double* fine, float* coarse) {
  k_restrict<<<nn_blocks(int64_t(Hc) * Wc, 256), 256, 0, c.stream>>>(Hc, Wc, 1 << levels, fine, coarse);
  after_launch(c, "grid_restrict");
}

void grid_prolong(Ctx& c, int Hc, int Wc, int levels, const float* coarse, double* fine) {
  const int64_t nc = int64_t(Hc) * Wc;
  if (levels == 0) {
    k_to_double<<<nn_blocks(nc, 256), 256, 0, c.stream>>>(nc, coarse, fine);
    after_launch(c, "grid_to_double");
    return;
  }
  // ping-pong buffers hold every level but the last (at most nc 4^(levels - 1) values)
  const size_t cap = size_t(nc) << (2 * (levels - 1));
  DBuf a(&c, cap), b(&c, cap);
  k_to_double<<<nn_blocks(nc, 256), 256, 0, c.stream>>>(nc, coarse, a.p);
  after_launch(c, "grid_to_double");
  int H = Hc, W = Wc;
  double* cur = a.p;
  for (int l = 0; l < levels; ++l) {
    double* out = (l == levels - 1) ? fine : (cur == a.p ? b.p : a.p);
    k_prolong2<<<nn_blocks(int64_t(4) * H * W, 256), 256, 0, c.stream>>>(H, W, cur, out);
    after_launch(c, "grid_prolong2");
    cur = out;
    H *= 2;
    W *= 2;
  }
}

void field_moments(Ctx& c, int64_t n, const float* x, double* out_dev) {
  k_moments<<<1, 1024, 0, c.stream>>>(n, x, out_dev);
  after_launch(c, "field_moments");
}

}  // namespace qtt

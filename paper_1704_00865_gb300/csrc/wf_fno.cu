// wf_fno.cu -- a Fourier neural operator (FNO) that predicts the Wiener
// solution from the data and noise weights, trained on the GPU with hand-
// written forward and backward kernels and Adam, and used to start the
// messenger iteration (the paper has no network; this is an extension).
//
// Network, for input x [B, 2, N, N] (data and log noise weight):
//   h_0 = P x + p;   h_{l+1} = act(W_l h_l + w_l + K_l h_l), l < L
//   (act = GELU, identity after the last layer);   y = Q h_L + q.
// K_l is the spectral convolution on the retained modes k_x in [0, MX),
// k_y in [0, MY) U [N - MY, N): a truncated real 2D DFT of each channel, one
// complex width x width matrix per mode, and the truncated inverse
// (1/N^2, real part, k_x > 0 counted twice).  The truncated transforms are
// direct sums with twiddle tables: for 16 x 32 retained modes that is fewer
// operations than a full FFT and needs no transpose.
//
// Layout: activations [B][C][N][N] FP32.  Weights live as an FP32 master
// vector (the order of the test oracle's flatten: P, p, per layer W_l, w_l,
// R_l as interleaved (re, im), then Q, q) with Adam moments; the forward and
// backward passes read an FP16 copy of the matrices (P, W_l, R_l, Q) and the
// FP32 biases, and accumulate in FP32.  Gradients are with respect to the
// FP16-rounded weights and update the FP32 master.  Every reduction runs in
// a fixed order (per-block partial sums, then one block), so a training
// step repeats bit for bit.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "../../include/wf.h"
#include "wf_device.cuh"
#include "wf_internal.h"

namespace {

constexpr int kThreads = 256;
constexpr int kMaxWidth = 64;
constexpr int kMaxModes = 32;

struct Layout {
  int cin = 2, width = 0, mx = 0, my = 0, layers = 0;
  size_t oP = 0, op = 0, oQ = 0, oq = 0, total = 0;
  std::vector<size_t> oW, ow, oR;
  void build() {
    size_t o = 0;
    oP = o; o += (size_t)width * cin;
    op = o; o += width;
    oW.resize(layers); ow.resize(layers); oR.resize(layers);
    for (int l = 0; l < layers; ++l) {
      oW[l] = o; o += (size_t)width * width;
      ow[l] = o; o += width;
      oR[l] = o; o += (size_t)width * width * 2 * my * mx * 2;
    }
    oQ = o; o += width;
    oq = o; o += 1;
    total = o;
  }
};

// ------------------------------------------------------------------ kernels

__global__ void to_half_kernel(const float* __restrict__ src, __half* __restrict__ dst, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    dst[i] = __float2half_rn(src[i]);
}

// The network's passes (sizes: B maps, C channels of N x N pixels, MX x 2 MY
// retained modes; CP = C rounded up to 8, 16, 32 or 64).
//
//   analysis     rows and columns of the truncated DFT of a block of rows of
//                one channel -> partial sums of X[j][k]
//   mix          the partial sums -> X; Y = R X (or R^H X for the adjoint)
//   synth_cols   Y -> S[y][k], the truncated inverse along columns
//   synth        S -> pixels along rows, + W h + bias, GELU (or the adjoint,
//                times GELU')
//
// A layer is four launches forward and seven backward; each activation map is
// read twice and written once.  Before, the transforms were one output per
// thread with both operands from L2, and the channel products kept their
// operands in local memory: inference of one 512^2 map (32 channels, 16 x 32
// modes, 4 layers) 6359 us then, 303 us now; the gradient of eight 256^2 maps
// 15 600 us then, 1340 us now.
//
// Both transforms use e^{2 pi i k (x + N/2) / N} = (-1)^k e^{2 pi i k x / N}: rows
// (and columns) a half period apart are added and subtracted first, the sums
// serve the even k and the differences the odd k, so every direct sum runs
// over N/2 terms (or gives two outputs).

constexpr int kAnRows = 64;   // rows of an analysis block, half of them N/2 further on
constexpr int kAnX = 32;      // pixels of a row staged at a time
constexpr int kMixModes = 8;  // modes of a mix block
constexpr int kColY = 32;     // row pairs of a column-synthesis block

// h_0 = P x + p
__global__ void lift_fwd(const float* __restrict__ x, const __half* __restrict__ W, const float* __restrict__ bias,
                         float* __restrict__ out, int B, int C, int P) {
  __shared__ float sW[kMaxWidth * 2];
  __shared__ float sb[kMaxWidth];
  for (int k = threadIdx.x; k < 2 * C; k += blockDim.x) sW[k] = __half2float(W[k]);
  for (int k = threadIdx.x; k < C; k += blockDim.x) sb[k] = bias[k];
  __syncthreads();
  const size_t total = (size_t)B * P;
  for (size_t g = blockIdx.x * (size_t)blockDim.x + threadIdx.x; g < total; g += (size_t)gridDim.x * blockDim.x) {
    const int b = (int)(g / P), p = (int)(g % P);
    const float x0 = x[((size_t)b * 2) * P + p], x1 = x[((size_t)b * 2 + 1) * P + p];
    for (int o = 0; o < C; ++o)
      out[((size_t)b * C + o) * P + p] = fmaf(sW[2 * o + 1], x1, fmaf(sW[2 * o], x0, sb[o]));
  }
}

// Partial column sums of the row DFTs of one channel's rows:
//   part[slice][block][j][k] = sc_k sum_{y in block} e^{-2 pi i ky_j y / N} sum_x in[y][x] e^{-2 pi i k x / N}
// for the 64 rows {y0 .. y0 + 31} and the same + N/2.  The row DFT is a
// register-tiled product of the folded rows with the twiddle table
// tw_k[x][parity][mode]: a warp takes eight modes of one parity for all rows, a
// lane two rows, so the twiddles are the same for the whole warp (broadcast
// loads) and a step is 32 FMA for one 8-byte and four broadcast 16-byte loads
// (with 4 rows x 2 modes a thread, both operands lane-dependent, the shared
// loads took twice the FMA's time: 42 us for eight 256^2 maps of 32 channels).
// The folded rows are staged transposed, row groups XOR-swizzled by x so that
// the stores are conflict-free.  KS groups of warps share the pixels of a row
// (each with its own stage and its own barrier) so that few rows still fill
// the SMs; their sums (of N / (2 KS) terms: 128 at 1024^2 with four groups, up
// to 512 with one) are added in a fixed order.  FP32 bound: N/2 * 32 FMA per row
// for 16 modes.
template <int KS, int KW>
__global__ void __launch_bounds__(KS * KW * 64, KW == 1 ? (KS == 4 ? 3 : 10) : 1)
analysis(const float* __restrict__ in, float2* __restrict__ part, const float2* __restrict__ tw_k,
         const float2* __restrict__ tw_y, int N, int MX, int MY2, float s0, float s1) {
  extern __shared__ __align__(16) float sm_an[];
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  const int GW = 2 * KW;                              // warps of a group: KW sets of 8 modes per parity
  const int gt = GW * 32, grp = tid / gt, gtid = tid - grp * gt, gw = gtid >> 5;
  const int rows = min(kAnRows, N), RH = rows / 2, nblk = (N / 2) / RH;
  const int slice = blockIdx.x / nblk, yb = blockIdx.x - slice * nblk;
  const int y0 = yb * RH;
  const int lx = min(5, 31 - __clz(N / 2)), NX = 1 << lx;  // pixels staged at a time
  const size_t gsz = 2 * kAnX * kAnRows + kAnX * 2 * KW * 16;
  float* st = sm_an + grp * gsz;                      // [2][kAnX][kAnRows] folded rows
  float4* stw = reinterpret_cast<float4*>(st + 2 * kAnX * kAnRows);  // [kAnX][2 KW][4] mode pairs
  const float* src = in + (size_t)slice * N * N;
  const int par = gw >= KW ? 1 : 0;
  float acc[2][16];                                   // [row][mode, re / im]
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int q = 0; q < 16; ++q) acc[r][q] = 0.f;
  const int pieces = rows << (lx - 2);                // 16-byte pieces of the stage
  for (int x0 = grp * NX; x0 < N / 2; x0 += KS * NX) {
    asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(gt) : "memory");
    for (int i = gtid; i < pieces; i += gt) {
      const int r4 = i & 3, xq = (i >> 2) & ((NX >> 2) - 1), rq = i >> lx;
      const int row = rq * 4 + r4;
      const int y = row < RH ? y0 + row : y0 + N / 2 + row - RH;
      const float4 a = *reinterpret_cast<const float4*>(src + (size_t)y * N + x0 + 4 * xq);
      const float4 b = *reinterpret_cast<const float4*>(src + (size_t)y * N + x0 + N / 2 + 4 * xq);
      float* d = st + (4 * xq) * kAnRows + ((rq ^ (xq & 7)) * 4 + r4);
      d[0] = a.x + b.x;
      d[kAnRows] = a.y + b.y;
      d[2 * kAnRows] = a.z + b.z;
      d[3 * kAnRows] = a.w + b.w;
      d += kAnX * kAnRows;
      d[0] = a.x - b.x;
      d[kAnRows] = a.y - b.y;
      d[2 * kAnRows] = a.z - b.z;
      d[3 * kAnRows] = a.w - b.w;
    }
    for (int i = gtid; i < NX * 2 * KW * 4; i += gt)
      stw[i] = __ldg(reinterpret_cast<const float4*>(tw_k) + (size_t)x0 * 2 * KW * 4 + i);
    asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(gt) : "memory");
    const float* sp = st + par * kAnX * kAnRows + 2 * (lane & 1);
    const float4* wp = stw + gw * 4;
#pragma unroll 4
    for (int x = 0; x < NX; ++x) {
      const float2 h = *reinterpret_cast<const float2*>(sp + x * kAnRows + (((lane >> 1) ^ ((x >> 2) & 7)) * 4));
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 w = wp[x * 2 * KW * 4 + q];
        const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc[0][4 * q + e] = fmaf(h.x, wv[e], acc[0][4 * q + e]);
          acc[1][4 * q + e] = fmaf(h.y, wv[e], acc[1][4 * q + e]);
        }
      }
    }
  }
  // the row transforms [MX][RS], the groups' shares added one after another
  float2* sA = reinterpret_cast<float2*>(sm_an);
  const int RS = rows + 1;
  for (int g = 0; g < KS; ++g) {
    __syncthreads();
    if (grp == g) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int k = 2 * (8 * (gw - par * KW) + q) + par;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int row = 2 * lane + r;
          if (k < MX && row < rows) {
            float2 v = make_float2(acc[r][2 * q], acc[r][2 * q + 1]);
            if (g > 0) {
              const float2 o = sA[k * RS + row];
              v = make_float2(v.x + o.x, v.y + o.y);
            }
            if (g == KS - 1) {
              const float sc = k == 0 ? s0 : s1;
              v = make_float2(v.x * sc, v.y * sc);
            }
            sA[k * RS + row] = v;
          }
        }
      }
    }
  }
  __syncthreads();
  for (int i = tid; i < RH * MX; i += nt) {  // fold the rows a half period apart
    float2* c = sA + (i / RH) * RS + (i % RH);
    const float2 a = c[0], b = c[RH];
    c[0] = make_float2(a.x + b.x, a.y + b.y);
    c[RH] = make_float2(a.x - b.x, a.y - b.y);
  }
  __syncthreads();
  // the block's share of the columns, JQ k_y of one parity (ky_j has the
  // parity of j: N - 2 MY is even) per thread
  constexpr int JQ = KS == 4 ? 2 : 4;
  float2* dst = part + ((size_t)slice * nblk + yb) * MY2 * MX;
  const int MY = MY2 / 2, JG = (MY + JQ - 1) / JQ;
  for (int i = tid; i < 2 * JG * MX; i += nt) {
    const int k = i % MX, pj = i / MX, pa = pj & 1, j0 = 2 * JQ * (pj >> 1) + pa;
    const float2* a = sA + k * RS + pa * RH;
    const float2* w[JQ];
    float re[JQ], im[JQ];
#pragma unroll
    for (int q = 0; q < JQ; ++q) {
      w[q] = tw_y + (size_t)min(j0 + 2 * q, MY2 - 1) * N + y0;
      re[q] = im[q] = 0.f;
    }
#pragma unroll 8
    for (int y = 0; y < RH; ++y) {
      const float2 v = a[y];
#pragma unroll
      for (int q = 0; q < JQ; ++q) {
        const float2 t = __ldg(&w[q][y]);
        re[q] = fmaf(v.x, t.x, fmaf(-v.y, t.y, re[q]));
        im[q] = fmaf(v.x, t.y, fmaf(v.y, t.x, im[q]));
      }
    }
#pragma unroll
    for (int q = 0; q < JQ; ++q)
      if (j0 + 2 * q < MY2) dst[(j0 + 2 * q) * MX + k] = make_float2(re[q], im[q]);
  }
}

// X[b][c][m] = the sum of the blocks' partial sums; then, per mode m,
//   fwd: out[b][m][o] = sum_i R[i][o][m] X[b][i][m]
//   bwd: out[b][m][i] = sum_o conj(R[i][o][m]) X[b][o][m]
// One block takes 8 modes (32-byte pieces of R) of one map; the output is
// channel-fastest for the column synthesis.  Bound by the latency of reading R
// (4 C^2 bytes per mode): two halves of the block share the summed channels and
// keep 16 loads each in flight.
__global__ void __launch_bounds__(2 * kThreads)
mix(const float2* __restrict__ part, int nblk, const __half2* __restrict__ R, float2* __restrict__ X,
    float2* __restrict__ out, int C, int CP, int NM, int bwd) {
  __shared__ float2 sX[kMaxWidth * kMixModes];
  __shared__ float2 sY[2][kMixModes * kMaxWidth];
  const int b = blockIdx.y, m0 = blockIdx.x * kMixModes;
  const int half = threadIdx.x / kThreads, c0 = half * (C / 2), c1 = half ? C : C / 2;  // C is even
  const int i0 = threadIdx.x % kThreads;
  const size_t rs = bwd ? (size_t)NM : (size_t)C * NM, ro = bwd ? (size_t)C * NM : (size_t)NM;
  // the first 16 matrix values of the first output, before the sums
  __half2 rv[16];
  {
    const int o = i0 / kMixModes, m = m0 + i0 % kMixModes;
#pragma unroll
    for (int q = 0; q < 16; ++q)
      rv[q] = (o < C && m < NM && c0 + q < c1) ? R[(size_t)o * ro + (size_t)(c0 + q) * rs + m] : __half2();
  }
  for (int i = threadIdx.x; i < C * kMixModes; i += blockDim.x) {
    const int c = i / kMixModes, m = m0 + i % kMixModes;
    float re = 0.f, im = 0.f;
    if (m < NM) {
      const float2* src = part + ((size_t)(b * C + c) * nblk) * NM + m;
#pragma unroll 8
      for (int q = 0; q < nblk; ++q) {
        const float2 v = src[(size_t)q * NM];
        re += v.x;
        im += v.y;
      }
      X[((size_t)b * C + c) * NM + m] = make_float2(re, im);
    }
    sX[i] = make_float2(re, im);
  }
  __syncthreads();
  const float sg = bwd ? -1.f : 1.f;  // conj(R) in the adjoint
  for (int i = i0; i < CP * kMixModes; i += kThreads) {
    const int o = i / kMixModes, ml = i % kMixModes, m = m0 + ml;
    float re = 0.f, im = 0.f;
    if (o < C && m < NM) {
      for (int cb = c0; cb < c1; cb += 16) {
        if (i != i0 || cb != c0) {
#pragma unroll
          for (int q = 0; q < 16; ++q)
            rv[q] = cb + q < c1 ? R[(size_t)o * ro + (size_t)(cb + q) * rs + m] : __half2();
        }
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          if (cb + q < c1) {
            const float2 r = __half22float2(rv[q]);
            const float2 x = sX[(cb + q) * kMixModes + ml];
            const float ry = sg * r.y;
            re = fmaf(r.x, x.x, fmaf(-ry, x.y, re));
            im = fmaf(r.x, x.y, fmaf(ry, x.x, im));
          }
        }
      }
    }
    sY[half][ml * CP + o] = make_float2(re, im);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < CP * kMixModes; i += blockDim.x) {
    const int m = m0 + i / CP;
    const float2 u = sY[0][i], v = sY[1][i];
    if (m < NM) out[((size_t)b * NM + m) * CP + i % CP] = make_float2(u.x + v.x, u.y + v.y);
  }
}

// g_R[i][o][m] = sum_b g_Y[b][o][m] conj(X[b][i][m]), written as (re, im)
// pairs: 4 x 4 channels of one mode per thread.  The bias gradient of the
// pointwise branch, the sum of g_z over all pixels, is N^2 times the mode 0
// of g_Y (scale 1/N^2 there): written by the threads of mode 0.
__global__ void __launch_bounds__(128)
mix_bwd_r(const float2* __restrict__ gY, const float2* __restrict__ X, float* __restrict__ gR, float* __restrict__ gw,
          int B, int C, int NM, float n2) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= NM) return;
  const int i0 = blockIdx.y * 4, o0 = blockIdx.z * 4;
  float re[4][4], im[4][4], bias[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int o = 0; o < 4; ++o) re[i][o] = im[i][o] = 0.f;
#pragma unroll 4
  for (int b = 0; b < B; ++b) {
    float2 x[4], y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      x[i] = i0 + i < C ? X[((size_t)b * C + i0 + i) * NM + m] : make_float2(0.f, 0.f);
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      y[o] = o0 + o < C ? gY[((size_t)b * C + o0 + o) * NM + m] : make_float2(0.f, 0.f);
      bias[o] += y[o].x;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        re[i][o] = fmaf(y[o].x, x[i].x, fmaf(y[o].y, x[i].y, re[i][o]));
        im[i][o] = fmaf(y[o].y, x[i].x, fmaf(-y[o].x, x[i].y, im[i][o]));
      }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int o = 0; o < 4; ++o)
      if (i0 + i < C && o0 + o < C) {
        // 8-byte aligned: widths are even, so every block of the vector is
        reinterpret_cast<float2*>(gR)[((size_t)(i0 + i) * C + o0 + o) * NM + m] = make_float2(re[i][o], im[i][o]);
      }
  if (m == 0 && i0 == 0)
#pragma unroll
    for (int o = 0; o < 4; ++o)
      if (o0 + o < C) gw[o0 + o] = bias[o] * n2;
}

// S[b][y][k] = c_k sum_j Y[b][j k] e^{+2 pi i ky_j y / N} for all channels, as
// CP real parts then CP imaginary parts (the imaginary part of k = 0 drops
// out of the row synthesis and is written as 0).  A lane is a channel, a warp
// takes four rows and, from the same sums, the four N/2 further on.
__global__ void __launch_bounds__(256)
synth_cols(const float2* __restrict__ Y, float* __restrict__ S, const float2* __restrict__ tw_y, int N, int MX,
           int MY2, int CP, float c0, float c1) {
  extern __shared__ __align__(16) float2 sm_sc[];
  float2* sT = sm_sc;                  // [MY2][kColY]
  float2* sY = sm_sc + MY2 * kColY;    // [MY2][CP]
  const int yb = blockIdx.x * kColY, k = blockIdx.y, b = blockIdx.z;
  for (int i = threadIdx.x; i < MY2 * kColY; i += blockDim.x) {
    const int y = yb + i % kColY;
    sT[i] = y < N / 2 ? __ldg(&tw_y[(size_t)(i / kColY) * N + y]) : make_float2(0.f, 0.f);
  }
  for (int i = threadIdx.x; i < MY2 * CP; i += blockDim.x)
    sY[i] = Y[((size_t)b * MY2 * MX + (size_t)(i / CP) * MX + k) * CP + i % CP];
  __syncthreads();
  const int lane = threadIdx.x & 31, yl = (threadIdx.x >> 5) * 4;
  const float sc = k == 0 ? c0 : c1;
  for (int o = lane; o < CP; o += 32) {
    float er[4], ei[4], dr[4], di[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) er[q] = ei[q] = dr[q] = di[q] = 0.f;
    for (int j = 0; j < MY2; j += 2) {
      const float2 a = sY[j * CP + o], c = sY[(j + 1) * CP + o];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float2 t = sT[j * kColY + yl + q], u = sT[(j + 1) * kColY + yl + q];  // conjugates of e^{+...}
        er[q] = fmaf(a.x, t.x, fmaf(a.y, t.y, er[q]));
        ei[q] = fmaf(-a.x, t.y, fmaf(a.y, t.x, ei[q]));
        dr[q] = fmaf(c.x, u.x, fmaf(c.y, u.y, dr[q]));
        di[q] = fmaf(-c.x, u.y, fmaf(c.y, u.x, di[q]));
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int y = yb + yl + q;
      if (y < N / 2) {
        float* d = S + (((size_t)b * N + y) * MX + k) * 2 * CP + o;
        d[0] = (er[q] + dr[q]) * sc;
        d[CP] = k == 0 ? 0.f : (ei[q] + di[q]) * sc;
        d += (size_t)(N / 2) * MX * 2 * CP;
        d[0] = (er[q] - dr[q]) * sc;
        d[CP] = k == 0 ? 0.f : (ei[q] - di[q]) * sc;
      }
    }
  }
}

// packed FP32 pairs (low word first)
__device__ __forceinline__ unsigned long long pack2(float x, float y) {
  return (unsigned long long)__float_as_uint(x) | ((unsigned long long)__float_as_uint(y) << 32);
}
__device__ __forceinline__ unsigned long long dup2(float x) { return pack2(x, x); }
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  return make_float2(__uint_as_float((unsigned)v), __uint_as_float((unsigned)(v >> 32)));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// Geometry of the row synthesis: OG groups of 8 output channels x PG groups
// of 2 pixel pairs (x, x + N/2); XT pairs of one row, RT rows per step.
__host__ __device__ constexpr int synth_pg(int OG) { return 256 / OG < 64 ? 256 / OG : 64; }
struct SynthGeom {
  int XT, RT, nxt, units;
  size_t smem;
};
inline SynthGeom synth_geom(int OG, int B, int C, int N, int MX) {
  SynthGeom g;
  const int pairs = 2 * synth_pg(OG);
  g.XT = N / 2 < pairs ? N / 2 : pairs;
  g.RT = pairs / g.XT < 4 ? pairs / g.XT : 4;
  g.nxt = (N / 2) / g.XT;
  g.units = B * (N / g.RT) * g.nxt;
  const int CP = 8 * OG;
  g.smem = sizeof(float) * ((size_t)C * CP + (size_t)2 * MX * g.XT +
                            2 * ((size_t)g.RT * MX * 2 * CP + (size_t)C * 2 * g.RT * g.XT));
  return g;
}

struct SynthArgs {
  const float* in;     // [B][C][N][N]: h_l (forward) or g_z (adjoint)
  const __half* W;     // [C][C]
  const float* S;      // [B][N][MX][2][CP]
  const float2* tw_x;  // [MX][N]
  const float* bias;   // forward
  float* out;          // or nullptr
  float* dact;         // forward: act'(z), or nullptr
  const float* mul;    // adjoint: act'(z) of the layer below, or nullptr
  const __half* Q;     // forward: project the output onto y, or nullptr
  const float* q;
  float* y;            // [B][N][N]
  const float* x;      // adjoint of layer 0: network input, for the lift's gradient, or nullptr
  float* lpart;        // [blocks][CP][3] sums of g x0, g x1, g
  int B, C, N, MX, XT, RT, nxt, units, act;
};

// One layer in pixels.  Forward: z = bias + W h + (row synthesis of S), out =
// act(z), act' kept for the backward pass (one erff serves both), the last
// layer projected onto y.  Adjoint (ADJ): g = W^T g_z + (row synthesis of S),
// times act' of the layer below; for layer 0 the sums of the lift's
// gradient instead.  A thread holds 8 channels x 4 pixels (two neighbours and
// the two N/2 further on); a warp has one channel group, so its weights and
// modes are broadcast loads and its pixel loads and stores are whole lines.
// The channels go in pairs through the packed FP32 FMA: the pairs are the
// registers a 16-byte load of the weights gives, only the pixel value is
// duplicated, and a step of 32 FMA issues 16 FMA, 4 moves and 4 loads.  The
// tables (W, the row twiddles of the block's pixels) stay in shared memory
// while the block walks its rows.  1536 FMA per pixel at 32 channels and 16
// modes (FP32 bound, 21 us for eight 256^2 maps) against 8 to 12 C bytes: 69
// us measured, about a fifth of it the erf; with the channel groups across the
// lanes of a warp, scalar FMA and one stage it took 93 us.
template <int OG, bool ADJ, bool FULL>
__global__ void __launch_bounds__(OG * synth_pg(OG))
synth(SynthArgs a) {
  constexpr int PG = synth_pg(OG), NT = OG * PG, CP = 8 * OG;
  extern __shared__ __align__(16) float sm_sy[];
  // FULL: the channels fill their groups and a step is part of one row, so
  // the strides and loop bounds are known
  const int N = a.N, MX = a.MX;
  const int C = FULL ? CP : a.C, XT = FULL ? 2 * PG : a.XT, RT = FULL ? 1 : a.RT, PX = RT * XT;
  const size_t P = (size_t)N * N;
  float* sW = sm_sy;                                 // [C][CP]: input channel, output channel
  float* sTc = sW + (size_t)C * CP;                  // [MX][XT] cos
  float* sTs = sTc + (size_t)MX * XT;                // [MX][XT] -sin
  float* sStage = sTs + (size_t)MX * XT;             // two stages of:
  const size_t szS = (size_t)RT * MX * 2 * CP;       // S  [RT][MX][2][CP]
  const size_t szStage = szS + (size_t)C * 2 * PX;   // h  [C][2][RT][XT]
  const int tid = threadIdx.x, og = (tid >> 5) % OG, pg = (tid & 31) + 32 * ((tid >> 5) / OG);
  const int xt = blockIdx.x % a.nxt;                 // gridDim.x is a multiple of nxt
  for (int i = tid; i < C * CP; i += NT) {
    const int ci = i / CP, co = i % CP;
    sW[i] = co < C ? __half2float(ADJ ? a.W[ci * C + co] : a.W[co * C + ci]) : 0.f;
  }
  for (int i = tid; i < MX * XT; i += NT) {
    const float2 t = __ldg(&a.tw_x[(size_t)(i / XT) * N + xt * XT + i % XT]);
    sTc[i] = t.x;
    sTs[i] = t.y;
  }
  const int pr = 2 * pg;                             // this thread's first pair
  const bool on = FULL || pr < PX;
  const int rl = FULL || !on ? 0 : pr / XT, xl = FULL ? pr : (on ? pr % XT : 0);
  float bias[8], lsum[8][3];
#pragma unroll
  for (int o = 0; o < 8; ++o) {
    bias[o] = (!ADJ && og * 8 + o < C) ? a.bias[og * 8 + o] : 0.f;
    lsum[o][0] = lsum[o][1] = lsum[o][2] = 0.f;
  }
  const int nyb = N / RT;
  const int lxq = 31 - __clz(XT / 4), lrt = 31 - __clz(RT);  // powers of two
  auto stage = [&](int u, int st) {
    if (u < a.units) {
      const int t = u / a.nxt, y0 = (t % nyb) * RT, b = t / nyb;
      float* dS = sStage + st * szStage;
      float* dH = dS + szS;
      for (int i = tid; i < C << (lxq + lrt + 1); i += NT) {
        const int xq = i & ((1 << lxq) - 1), r = (i >> lxq) & (RT - 1), h = (i >> (lxq + lrt)) & 1,
                  c = i >> (lxq + lrt + 1);
        wf::cp_async16(dH + 4 * (size_t)i,
                       a.in + ((size_t)b * C + c) * P + (size_t)(y0 + r) * N + h * (N / 2) + xt * XT + 4 * xq);
      }
      const float* gs = a.S + ((size_t)b * N + y0) * MX * 2 * CP;
      for (int i = tid; i < (int)(szS / 4); i += NT) wf::cp_async16(dS + 4 * i, gs + 4 * i);
    }
    wf::cp_async_commit();
  };
  stage(blockIdx.x, 0);
  int cur = 0;
  for (int u = blockIdx.x; u < a.units; u += gridDim.x, cur ^= 1) {
    const int t = u / a.nxt, yb = t % nyb, b = t / nyb;
    const int y0 = yb * RT;
    // the stage filled next was read in the last step (barrier at its end)
    stage(u + gridDim.x, cur ^ 1);
    wf::cp_async_wait<1>();
    __syncthreads();
    const float* sS = sStage + cur * szStage;
    float* sH = sStage + cur * szStage + szS;
    // [channel pair][x, x + 1, x + N/2, x + N/2 + 1]
    unsigned long long zz[4][4];
#pragma unroll
    for (int o = 0; o < 4; ++o) zz[o][0] = zz[o][1] = zz[o][2] = zz[o][3] = 0ull;
    // modes: even k into [.][0..1], odd k into [.][2..3]
    const float* s = sS + (size_t)rl * MX * 2 * CP + og * 8;
#pragma unroll 2
    for (int k = 0; k < MX; k += 2) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (k + h < MX) {
          const float2 c = *reinterpret_cast<const float2*>(sTc + (k + h) * XT + xl);
          const float2 sn = *reinterpret_cast<const float2*>(sTs + (k + h) * XT + xl);
          const ulonglong2* sr = reinterpret_cast<const ulonglong2*>(s + (k + h) * 2 * CP);
          const ulonglong2* si = reinterpret_cast<const ulonglong2*>(s + (k + h) * 2 * CP + CP);
          const ulonglong2 r0 = sr[0], r1 = sr[1], i0 = si[0], i1 = si[1];
          const unsigned long long re[4] = {r0.x, r0.y, r1.x, r1.y}, im[4] = {i0.x, i0.y, i1.x, i1.y};
          const unsigned long long cx = dup2(c.x), cy = dup2(c.y), sx = dup2(sn.x), sy = dup2(sn.y);
#pragma unroll
          for (int o = 0; o < 4; ++o) {
            zz[o][2 * h] = fma2(re[o], cx, fma2(im[o], sx, zz[o][2 * h]));
            zz[o][2 * h + 1] = fma2(re[o], cy, fma2(im[o], sy, zz[o][2 * h + 1]));
          }
        }
      }
    }
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      float2 e0 = unpack2(zz[o][0]), e1 = unpack2(zz[o][1]), d0 = unpack2(zz[o][2]), d1 = unpack2(zz[o][3]);
      const float b0 = bias[2 * o], b1 = bias[2 * o + 1];
      zz[o][0] = pack2(e0.x + d0.x + b0, e0.y + d0.y + b1);
      zz[o][1] = pack2(e1.x + d1.x + b0, e1.y + d1.y + b1);
      zz[o][2] = pack2(e0.x - d0.x + b0, e0.y - d0.y + b1);
      zz[o][3] = pack2(e1.x - d1.x + b0, e1.y - d1.y + b1);
    }
    const float* hp = sH + (on ? pr : 0);
#pragma unroll 4
    for (int c = 0; c < C; ++c) {
      const float2 h0 = *reinterpret_cast<const float2*>(hp + (size_t)c * 2 * PX);
      const float2 h1 = *reinterpret_cast<const float2*>(hp + (size_t)c * 2 * PX + PX);
      const ulonglong2* wp = reinterpret_cast<const ulonglong2*>(sW + c * CP + og * 8);
      const ulonglong2 w0 = wp[0], w1 = wp[1];
      const unsigned long long w[4] = {w0.x, w0.y, w1.x, w1.y};
      const unsigned long long a0 = dup2(h0.x), a1 = dup2(h0.y), b0 = dup2(h1.x), b1 = dup2(h1.y);
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        zz[o][0] = fma2(w[o], a0, zz[o][0]);
        zz[o][1] = fma2(w[o], a1, zz[o][1]);
        zz[o][2] = fma2(w[o], b0, zz[o][2]);
        zz[o][3] = fma2(w[o], b1, zz[o][3]);
      }
    }
    __syncthreads();  // the tile is read: the next step's copies may overwrite it
    float z[8][4];
#pragma unroll
    for (int o = 0; o < 4; ++o)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 v = unpack2(zz[o][e]);
        z[2 * o][e] = v.x;
        z[2 * o + 1][e] = v.y;
      }
    const size_t px = (size_t)(y0 + rl) * N + xt * XT + xl;  // and px + N/2
    if constexpr (!ADJ) {
      float yv[4] = {0.f, 0.f, 0.f, 0.f};
      if (on) {
#pragma unroll
        for (int o = 0; o < 8; ++o) {
          const int co = og * 8 + o;
          if (co < C) {
            const size_t idx = ((size_t)b * C + co) * P + px;
            if (a.Q) {
              const float qv = __half2float(a.Q[co]);
#pragma unroll
              for (int e = 0; e < 4; ++e) yv[e] = fmaf(qv, z[o][e], yv[e]);
            }
            if (a.act) {
              float g[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const float v = z[o][e];
                const float Phi = 0.5f * (1.f + erff(v * 0.70710678118654752f));
                // d/dz [z Phi(z)] = Phi(z) + z phi(z)
                if (a.dact) g[e] = fmaf(v, 0.3989422804014327f * __expf(-0.5f * v * v), Phi);
                z[o][e] = v * Phi;
              }
              if (a.dact) {
                *reinterpret_cast<float2*>(a.dact + idx) = make_float2(g[0], g[1]);
                *reinterpret_cast<float2*>(a.dact + idx + N / 2) = make_float2(g[2], g[3]);
              }
            }
            if (a.out) {
              *reinterpret_cast<float2*>(a.out + idx) = make_float2(z[o][0], z[o][1]);
              *reinterpret_cast<float2*>(a.out + idx + N / 2) = make_float2(z[o][2], z[o][3]);
            }
          }
        }
      }
      if (a.Q) {  // sum the channel groups (the warps of these pixels) in order
        if (on) *reinterpret_cast<float4*>(sH + (og * PG + pg) * 4) = make_float4(yv[0], yv[1], yv[2], yv[3]);
        __syncthreads();
        if (on && og == 0) {
#pragma unroll
          for (int g = 1; g < OG; ++g) {
            const float4 v = *reinterpret_cast<const float4*>(sH + (g * PG + pg) * 4);
            yv[0] += v.x;
            yv[1] += v.y;
            yv[2] += v.z;
            yv[3] += v.w;
          }
          float* yo = a.y + (size_t)b * P + px;
          const float q = a.q[0];
          yo[0] = yv[0] + q;
          yo[1] = yv[1] + q;
          yo[N / 2] = yv[2] + q;
          yo[N / 2 + 1] = yv[3] + q;
        }
        __syncthreads();
      }
    } else if (on) {
      float xv[2][4];
      if (a.x) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float* xp = a.x + ((size_t)b * 2 + i) * P + px;
          xv[i][0] = xp[0];
          xv[i][1] = xp[1];
          xv[i][2] = xp[N / 2];
          xv[i][3] = xp[N / 2 + 1];
        }
      }
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        const int co = og * 8 + o;
        if (co < C) {
          const size_t idx = ((size_t)b * C + co) * P + px;
          if (a.mul) {
            const float2 g0 = *reinterpret_cast<const float2*>(a.mul + idx);
            const float2 g1 = *reinterpret_cast<const float2*>(a.mul + idx + N / 2);
            z[o][0] *= g0.x;
            z[o][1] *= g0.y;
            z[o][2] *= g1.x;
            z[o][3] *= g1.y;
          }
          if (a.out) {
            *reinterpret_cast<float2*>(a.out + idx) = make_float2(z[o][0], z[o][1]);
            *reinterpret_cast<float2*>(a.out + idx + N / 2) = make_float2(z[o][2], z[o][3]);
          }
          if (a.x) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
              lsum[o][i] += fmaf(z[o][0], xv[i][0], z[o][1] * xv[i][1]) +
                            fmaf(z[o][2], xv[i][2], z[o][3] * xv[i][3]);
            lsum[o][2] += (z[o][0] + z[o][1]) + (z[o][2] + z[o][3]);
          }
        }
      }
    }
  }
  if constexpr (ADJ) {
    if (a.x) {  // the block's sums over its pixels: a fixed tree
      wf::cp_async_wait<0>();
      __syncthreads();
#pragma unroll
      for (int o = 0; o < 8; ++o)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          float v = lsum[o][i];
#pragma unroll
          for (int sft = 16; sft > 0; sft >>= 1) v += __shfl_xor_sync(0xffffffffu, v, sft);
          lsum[o][i] = v;
        }
      float* red = sm_sy;  // [warps][8][3] over the tables, which are done with
      if ((tid & 31) == 0)
#pragma unroll
        for (int o = 0; o < 8; ++o)
#pragma unroll
          for (int i = 0; i < 3; ++i) red[((tid >> 5) * 8 + o) * 3 + i] = lsum[o][i];
      __syncthreads();
      for (int i = tid; i < CP * 3; i += NT) {
        float v = 0.f;  // channel i / 3: the warps of group (i / 3) / 8
        for (int w = i / 24; w < NT / 32; w += OG) v += red[w * 24 + i % 24];
        a.lpart[(size_t)blockIdx.x * CP * 3 + i] = v;
      }
    }
  }
}

// partial[blk][o][i] = sum over this block's pixels of gz[b][o][p] in[b][i][p]:
// tiles of 128 pixels of all channels in shared memory (rows 4 floats apart
// in banks), 4 x 4 channels per thread, the pixels of a tile split over the
// 256 / (CP/4)^2 thread groups, whose sums are added in a fixed order.  Each
// tile is summed by itself and then added up.  C^2 FMA per pixel against 8 C
// bytes.
constexpr int kWgPx = 128, kWgStride = kWgPx + 4;
template <int CP>
__global__ void __launch_bounds__(256)
weight_grad(const float* __restrict__ gz, const float* __restrict__ in, float* __restrict__ partial, int B, int C,
            int P) {
  constexpr int G = CP / 4, GT = G * G;
  constexpr int SPLITS = 256 / GT < 32 ? 256 / GT : 32;  // at most one per 16-byte piece of a tile
  extern __shared__ __align__(16) float sm_wg[];  // two stages of a g and an h tile
  const int tid = threadIdx.x, grp = tid % GT, sp = tid / GT;
  const int og = grp / G, ig = grp % G;
  const bool on = sp < SPLITS;
  const int tiles_b = P / kWgPx, tiles = B * tiles_b;  // P = N^2 >= 256, a power of two
  float tot[4][4];
#pragma unroll
  for (int o = 0; o < 4; ++o)
#pragma unroll
    for (int i = 0; i < 4; ++i) tot[o][i] = 0.f;
  for (int c = C; c < CP; ++c)
    for (int x = tid; x < kWgPx; x += blockDim.x)
#pragma unroll
      for (int q = 0; q < 4; ++q) sm_wg[(q * CP + c) * kWgStride + x] = 0.f;
  auto stage = [&](int t, int st) {
    if (t < tiles) {
      const int b = t / tiles_b, p0 = (t - b * tiles_b) * kWgPx;
      float* d = sm_wg + 2 * st * CP * kWgStride;
      for (int i = tid; i < C * (kWgPx / 4); i += 256) {
        const int c = i / (kWgPx / 4), xq = i % (kWgPx / 4);
        const size_t o = ((size_t)b * C + c) * P + p0 + 4 * xq;
        wf::cp_async16(d + c * kWgStride + 4 * xq, gz + o);
        wf::cp_async16(d + (CP + c) * kWgStride + 4 * xq, in + o);
      }
    }
    wf::cp_async_commit();
  };
  stage(blockIdx.x, 0);
  int st = 0;
  for (int t = blockIdx.x; t < tiles; t += gridDim.x, st ^= 1) {
    stage(t + gridDim.x, st ^ 1);
    wf::cp_async_wait<1>();
    __syncthreads();
    if (on) {
      const float* sg = sm_wg + 2 * st * CP * kWgStride;
      const float* sh = sg + CP * kWgStride;
      float acc[4][4];
#pragma unroll
      for (int o = 0; o < 4; ++o)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[o][i] = 0.f;
      for (int xq = sp; xq < kWgPx / 4; xq += SPLITS) {
        float4 g[4], h[4];
#pragma unroll
        for (int o = 0; o < 4; ++o) g[o] = *reinterpret_cast<const float4*>(sg + (og + G * o) * kWgStride + 4 * xq);
#pragma unroll
        for (int i = 0; i < 4; ++i) h[i] = *reinterpret_cast<const float4*>(sh + (ig + G * i) * kWgStride + 4 * xq);
#pragma unroll
        for (int o = 0; o < 4; ++o)
#pragma unroll
          for (int i = 0; i < 4; ++i)
            acc[o][i] = fmaf(g[o].w, h[i].w, fmaf(g[o].z, h[i].z, fmaf(g[o].y, h[i].y, fmaf(g[o].x, h[i].x, acc[o][i]))));
      }
#pragma unroll
      for (int o = 0; o < 4; ++o)
#pragma unroll
        for (int i = 0; i < 4; ++i) tot[o][i] += acc[o][i];
    }
    __syncthreads();  // the stage is read before it is filled again
  }
  wf::cp_async_wait<0>();
  __syncthreads();
  float* red = sm_wg;  // [SPLITS][CP][CP]: at most 2 CP kWgStride floats (checked below)
  static_assert((CP >= 32 ? SPLITS : 8) * CP * CP <= 2 * CP * kWgStride, "reduction fits the tiles");
  constexpr int RS = (CP >= 32) ? SPLITS : 8;  // splits reduced at a time
  float sum[(CP * CP + 255) / 256];
#pragma unroll
  for (int q = 0; q < (CP * CP + 255) / 256; ++q) sum[q] = 0.f;
  for (int s0 = 0; s0 < SPLITS; s0 += RS) {
    if (on && sp >= s0 && sp < s0 + RS)
#pragma unroll
      for (int o = 0; o < 4; ++o)
#pragma unroll
        for (int i = 0; i < 4; ++i) red[((sp - s0) * CP + og + G * o) * CP + ig + G * i] = tot[o][i];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < (CP * CP + 255) / 256; ++q) {
      const int k = tid + 256 * q;
      if (k < CP * CP)
        for (int s = 0; s < RS; ++s) sum[q] += red[s * CP * CP + k];
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < (CP * CP + 255) / 256; ++q) {
    const int k = tid + 256 * q, o = k / CP, i = k % CP;
    if (k < CP * CP && o < C && i < C) partial[((size_t)blockIdx.x * C + o) * C + i] = sum[q];
  }
}

// Sums of nblk partial vectors of n values, a lane per value and 32 partial
// sums per value (fixed order).  map = 0:
// out[k]; map = 1: the lift's (o, {x0, x1, 1}) triples into gP [C][2] and gp
// [C]; map = 2: C values into out, then one into out2.
__global__ void __launch_bounds__(1024)
sum_partials(const float* __restrict__ partial, int nblk, int n, float* __restrict__ out, float* __restrict__ out2,
             int map, int C) {
  __shared__ float red[32][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int k = blockIdx.x * 32 + lane;
  float s = 0.f;
  if (k < n)
#pragma unroll 4
    for (int b = w; b < nblk; b += 32) s += partial[(size_t)b * n + k];
  red[w][lane] = s;
  __syncthreads();
  if (w != 0 || k >= n) return;
  s = 0.f;
#pragma unroll
  for (int i = 0; i < 32; ++i) s += red[i][lane];
  if (map == 0) {
    out[k] = s;
  } else if (map == 1) {
    const int o = k / 3, i = k % 3;
    if (o < C) {
      if (i < 2) out[o * 2 + i] = s;
      else out2[o] = s;
    }
  } else {
    if (k < C) out[k] = s;
    else if (k == n - 1) out2[0] = s;
  }
}

// Start of the backward pass: g_y = 2 (y - t) / (B ||t||^2), g_z of the last
// layer (no activation) = Q g_y, and the block's partial sums of the
// projection's gradient, g_y h_L and g_y ([blk][CP + 1]).  Bound by the latency
// of its loads: four blocks per SM (64 registers), 27 us for eight 256^2 maps of
// 32 channels against 43 us with two.
template <int CP>
__global__ void __launch_bounds__(kThreads, CP <= 32 ? 4 : 2)
proj_bwd(const float* __restrict__ y, const float* __restrict__ t, const float* __restrict__ inv,
         const __half* __restrict__ Q, const float* __restrict__ hL, float* __restrict__ gz, float* __restrict__ partial,
         int B, int C, int P) {
  __shared__ float sQ[CP];
  __shared__ float red[kThreads / 32][CP + 1];
  for (int i = threadIdx.x; i < CP; i += blockDim.x) sQ[i] = i < C ? __half2float(Q[i]) : 0.f;
  __syncthreads();
  float acc[CP], sg = 0.f;
#pragma unroll
  for (int o = 0; o < CP; ++o) acc[o] = 0.f;
  const size_t total = (size_t)B * P / 4;  // four pixels a step (P is a multiple of 256)
  for (size_t g = blockIdx.x * (size_t)blockDim.x + threadIdx.x; g < total; g += (size_t)gridDim.x * blockDim.x) {
    const size_t e = 4 * g;
    const int b = (int)(e / P);
    const float iv = inv[b];
    // t is the caller's: no alignment beyond a float's
    const float g0 = 2.f * (y[e] - t[e]) * iv, g1 = 2.f * (y[e + 1] - t[e + 1]) * iv,
                g2 = 2.f * (y[e + 2] - t[e + 2]) * iv, g3 = 2.f * (y[e + 3] - t[e + 3]) * iv;
    sg += (g0 + g1) + (g2 + g3);
    const size_t base = (size_t)b * C * P + (e - (size_t)b * P);
#pragma unroll
    for (int o = 0; o < CP; ++o)
      if (o < C) {
        const size_t idx = base + (size_t)o * P;
        const float4 h = *reinterpret_cast<const float4*>(hL + idx);
        acc[o] += fmaf(g0, h.x, g1 * h.y) + fmaf(g2, h.z, g3 * h.w);
        const float q = sQ[o];
        *reinterpret_cast<float4*>(gz + idx) = make_float4(q * g0, q * g1, q * g2, q * g3);
      }
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 0; o <= CP; ++o) {
    float v = o < CP ? acc[o < CP ? o : 0] : sg;
    for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
    if (lane == 0) red[w][o] = v;
  }
  __syncthreads();
  for (int o = threadIdx.x; o <= CP; o += blockDim.x) {
    float v = 0.f;
    for (int i = 0; i < kThreads / 32; ++i) v += red[i][o];
    partial[(size_t)blockIdx.x * (CP + 1) + o] = v;
  }
}

// per-sample sums of (y - t)^2 and t^2
__global__ void loss_partial(const float* __restrict__ y, const float* __restrict__ t, double* __restrict__ part,
                             int P) {
  const int b = blockIdx.y;
  double num = 0.0, den = 0.0;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < P; p += gridDim.x * blockDim.x) {
    const double d = (double)y[(size_t)b * P + p] - (double)t[(size_t)b * P + p];
    const double tv = t[(size_t)b * P + p];
    num += d * d;
    den += tv * tv;
  }
  __shared__ double rn[kThreads / 32], rd[kThreads / 32];
  for (int s = 16; s > 0; s >>= 1) {
    num += __shfl_xor_sync(0xffffffffu, num, s);
    den += __shfl_xor_sync(0xffffffffu, den, s);
  }
  if ((threadIdx.x & 31) == 0) {
    rn[threadIdx.x >> 5] = num;
    rd[threadIdx.x >> 5] = den;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, c = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      a += rn[w];
      c += rd[w];
    }
    part[((size_t)b * gridDim.x + blockIdx.x) * 2] = a;
    part[((size_t)b * gridDim.x + blockIdx.x) * 2 + 1] = c;
  }
}

// loss = mean_b num_b / den_b; inv[b] = 1 / (B den_b).  A warp per map: lane k
// sums block k (nblk = 32), then a fixed tree.
__global__ void loss_fin(const double* __restrict__ part, int nblk, int B, double* __restrict__ loss,
                         float* __restrict__ inv) {
  __shared__ double rel[64];  // B <= 64
  const int lane = threadIdx.x & 31;
  for (int b = threadIdx.x >> 5; b < B; b += blockDim.x >> 5) {
    double n = 0.0, d = 0.0;
    for (int k = lane; k < nblk; k += 32) {
      n += part[((size_t)b * nblk + k) * 2];
      d += part[((size_t)b * nblk + k) * 2 + 1];
    }
    for (int s = 16; s > 0; s >>= 1) {
      n += __shfl_xor_sync(0xffffffffu, n, s);
      d += __shfl_xor_sync(0xffffffffu, d, s);
    }
    d = d > 0.0 ? d : 1.0;
    if (lane == 0) {
      rel[b] = n / d;
      inv[b] = (float)(1.0 / (B * d));
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double L = 0.0;
    for (int b = 0; b < B; ++b) L += rel[b];
    *loss = L / B;
  }
}

__global__ void adam_kernel(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, size_t n, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// Inputs of the network for one map: x0 = d / sigma (0 on masked pixels),
// x1 = log(sigma^2 / pixel_var) (masked: log of a 1e-6 weight), with sigma^2
// the mean pixel variance over unmasked pixels (reduced in part/fin).
__global__ void feat_partial(const float* __restrict__ var, const uint8_t* __restrict__ mask, double* __restrict__ part,
                             size_t n) {
  double s = 0.0, c = 0.0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    if (mask && mask[i]) continue;
    s += var[i];
    c += 1.0;
  }
  __shared__ double rs[kThreads / 32], rc[kThreads / 32];
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    c += __shfl_xor_sync(0xffffffffu, c, o);
  }
  if ((threadIdx.x & 31) == 0) {
    rs[threadIdx.x >> 5] = s;
    rc[threadIdx.x >> 5] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      a += rs[w];
      b += rc[w];
    }
    part[2 * blockIdx.x] = a;
    part[2 * blockIdx.x + 1] = b;
  }
}

__global__ void feat_fin(const double* __restrict__ part, int nblk, float* __restrict__ sigma) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double a = 0.0, b = 0.0;
  for (int k = 0; k < nblk; ++k) {
    a += part[2 * k];
    b += part[2 * k + 1];
  }
  *sigma = (float)sqrt(b > 0.0 ? a / b : 1.0);
}

__global__ void feat_map(const float* __restrict__ d, const float* __restrict__ var, const uint8_t* __restrict__ mask,
                         const float* __restrict__ sigma, float* __restrict__ x, size_t n) {
  const float sg = *sigma;
  const float s2 = sg * sg;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const bool m = mask && mask[i];
    x[i] = m ? 0.f : d[i] / sg;
    x[n + i] = m ? logf(1e-6f) : logf(s2 / var[i]);
  }
}

int grid_for(size_t n) {
  const size_t g = (n + kThreads - 1) / kThreads;
  return (int)(g < 4096 ? (g > 0 ? g : 1) : 4096);
}

}  // namespace

struct wf_fno_s {
  Layout lay;
  int n = 0, batch = 0;
  cudaStream_t stream = nullptr;
  float *master = nullptr, *grad = nullptr, *m1 = nullptr, *m2 = nullptr;
  __half* half = nullptr;     // FP16 copy of the whole vector (matrices read from it)
  long long step = 0;
  // activations
  float* h = nullptr;         // [L+1][B][C][P]
  float* dact = nullptr;      // [L-1][B][C][P] GELU'(z) of the hidden layers
  float* y = nullptr;         // [B][P]
  float* gz = nullptr;        // [B][C][P] gradient wrt the current layer's z
  float2 *Xp = nullptr, *X = nullptr, *gY = nullptr, *Y = nullptr;  // partial sums, [L][B][C][2MY][MX], ...
  float* S = nullptr;         // [B][N][MX][2][CP]
  float2 *tw_x = nullptr, *tw_y = nullptr, *tw_k = nullptr;
  float* wpart = nullptr;
  int OG = 1, KW = 1, sms = 1, synth_per_sm = 1, adj_per_sm = 1;
  double* lpart = nullptr;
  double* dloss = nullptr;
  float* inv = nullptr;
  int lblk = 0;
  std::vector<void*> allocs;
};

namespace {

template <typename T>
bool alloc(wf_fno_s* F, T** p, size_t n) {
  if (cudaMalloc((void**)p, n * sizeof(T)) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  F->allocs.push_back(*p);
  return true;
}

size_t P_(const wf_fno_s* F) { return (size_t)F->n * F->n; }
size_t act_(const wf_fno_s* F) { return (size_t)F->batch * F->lay.width * P_(F); }
size_t modes_(const wf_fno_s* F) { return (size_t)2 * F->lay.my * F->lay.mx; }
int an_blocks(int n) { return (n / 2) / (std::min(kAnRows, n) / 2); }
size_t an_smem(int KS, int KW, int MX) {
  return sizeof(float) * std::max((size_t)KS * (2 * kAnX * kAnRows + kAnX * 2 * KW * 16), (size_t)2 * (kAnRows + 1) * MX);
}
size_t cols_smem(int MY2, int CP) { return sizeof(float2) * MY2 * (kColY + CP); }

// pixels or gradients [B][C][N][N] -> partial sums of the retained modes in Xp.
// Few blocks: four groups of warps each, from N = 256 on (every group then has
// its own 32 pixels of a half row): 26 us against 44 us for one 512^2 map of
// 32 channels (256 blocks).  From four blocks per SM on, one group, whose
// smaller stage lets more blocks share an SM: 39 us against 60 us for eight
// 256^2 maps (1024 blocks).
template <int KW>
void launch_analysis_kw(wf_fno_s* F, const float* in, int B, float s0, float s1) {
  const int C = F->lay.width, N = F->n, MX = F->lay.mx, MY2 = 2 * F->lay.my;
  const int grid = B * C * an_blocks(N);
  if (N >= 256 && grid < 4 * F->sms)
    analysis<4, KW><<<grid, 256 * KW, an_smem(4, KW, MX), F->stream>>>(in, F->Xp, F->tw_k, F->tw_y, N, MX, MY2, s0, s1);
  else
    analysis<1, KW><<<grid, 64 * KW, an_smem(1, KW, MX), F->stream>>>(in, F->Xp, F->tw_k, F->tw_y, N, MX, MY2, s0, s1);
}
void launch_analysis(wf_fno_s* F, const float* in, int B, float s0, float s1) {
  if (F->KW == 1) launch_analysis_kw<1>(F, in, B, s0, s1);
  else launch_analysis_kw<2>(F, in, B, s0, s1);
}

void launch_mix(wf_fno_s* F, int l, float2* X, int B, int bwd) {
  const int C = F->lay.width, NM = (int)modes_(F);
  const __half2* R = reinterpret_cast<const __half2*>(F->half + F->lay.oR[l]);
  mix<<<dim3((NM + kMixModes - 1) / kMixModes, B), 2 * kThreads, 0, F->stream>>>(F->Xp, an_blocks(F->n), R, X, F->Y, C,
                                                                             8 * F->OG, NM, bwd);
}

void launch_synth_cols(wf_fno_s* F, int B, float c0, float c1) {
  const int N = F->n, MX = F->lay.mx, MY2 = 2 * F->lay.my, CP = 8 * F->OG;
  synth_cols<<<dim3((N / 2 + kColY - 1) / kColY, MX, B), 256, cols_smem(MY2, CP), F->stream>>>(F->Y, F->S, F->tw_y, N,
                                                                                               MX, MY2, CP, c0, c1);
}

template <bool ADJ>
int synth_grid(const wf_fno_s* F, const SynthGeom& g) {
  // whole multiples of the pixel tiles of a row, at most one wave
  const int wave = F->sms * (ADJ ? F->adj_per_sm : F->synth_per_sm);
  const int n = std::min(g.units, wave);
  return std::max(g.nxt, n / g.nxt * g.nxt);
}

template <int OG, bool ADJ>
void launch_synth_og(wf_fno_s* F, const SynthArgs& a, const SynthGeom& g, int grid) {
  constexpr int nt = OG * synth_pg(OG);
  if (a.C == 8 * OG && g.RT == 1 && g.XT == 2 * synth_pg(OG)) synth<OG, ADJ, true><<<grid, nt, g.smem, F->stream>>>(a);
  else synth<OG, ADJ, false><<<grid, nt, g.smem, F->stream>>>(a);
}

template <bool ADJ>
int launch_synth(wf_fno_s* F, SynthArgs a, int B) {
  const SynthGeom g = synth_geom(F->OG, B, F->lay.width, F->n, F->lay.mx);
  a.B = B;
  a.C = F->lay.width;
  a.N = F->n;
  a.MX = F->lay.mx;
  a.XT = g.XT;
  a.RT = g.RT;
  a.nxt = g.nxt;
  a.units = g.units;
  a.S = F->S;
  a.tw_x = F->tw_x;
  const int grid = synth_grid<ADJ>(F, g);
  switch (F->OG) {
    case 1: launch_synth_og<1, ADJ>(F, a, g, grid); break;
    case 2: launch_synth_og<2, ADJ>(F, a, g, grid); break;
    case 4: launch_synth_og<4, ADJ>(F, a, g, grid); break;
    default: launch_synth_og<8, ADJ>(F, a, g, grid); break;
  }
  return grid;
}

// Blocks per SM of this network's synthesis (smem a block).  The limit belongs
// to the kernel on the device, not to the network: every network sets the same
// one, the most a block can have, or a network of a smaller footprint would
// take the launches of an earlier one away.
template <int OG, bool ADJ>
cudaError_t prepare_synth(size_t smem, int* per_sm) {
  int n0 = 0, n1 = 0;
  cudaError_t e =
      cudaFuncSetAttribute(synth<OG, ADJ, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wf::kMaxDynSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(synth<OG, ADJ, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wf::kMaxDynSmem);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n0, synth<OG, ADJ, false>, OG * synth_pg(OG), smem);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n1, synth<OG, ADJ, true>, OG * synth_pg(OG), smem);
  *per_sm = std::min(n0, n1);
  if (e == cudaSuccess && *per_sm < 1) e = cudaErrorInvalidConfiguration;
  return e;
}

constexpr size_t wg_smem(int CP) { return sizeof(float) * 4 * CP * kWgStride; }

// shared-memory sizes and blocks per SM of this network's kernels
cudaError_t prepare_kernels(wf_fno_s* F) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&F->sms, cudaDevAttrMultiProcessorCount, dev);
  const size_t sm = synth_geom(F->OG, 1, F->lay.width, F->n, F->lay.mx).smem;
  if (e == cudaSuccess) {
    switch (F->OG) {
      case 1: e = prepare_synth<1, false>(sm, &F->synth_per_sm); break;
      case 2: e = prepare_synth<2, false>(sm, &F->synth_per_sm); break;
      case 4: e = prepare_synth<4, false>(sm, &F->synth_per_sm); break;
      default: e = prepare_synth<8, false>(sm, &F->synth_per_sm); break;
    }
  }
  if (e == cudaSuccess) {
    switch (F->OG) {
      case 1: e = prepare_synth<1, true>(sm, &F->adj_per_sm); break;
      case 2: e = prepare_synth<2, true>(sm, &F->adj_per_sm); break;
      case 4: e = prepare_synth<4, true>(sm, &F->adj_per_sm); break;
      default: e = prepare_synth<8, true>(sm, &F->adj_per_sm); break;
    }
  }
  if (e == cudaSuccess && F->OG == 4)
    e = cudaFuncSetAttribute(weight_grad<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wg_smem(32));
  if (e == cudaSuccess && F->OG == 8)
    e = cudaFuncSetAttribute(weight_grad<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wg_smem(64));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(F->KW == 1 ? analysis<4, 1> : analysis<4, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)an_smem(4, F->KW, F->lay.mx));
  return e;
}

// the network on x into y (device); keep: the activations and act' of every
// layer stay for the backward pass
int forward(wf_fno_s* F, const float* x, float* y, int B, bool keep) {
  const Layout& L = F->lay;
  const int C = L.width, P = (int)P_(F);
  lift_fwd<<<grid_for((size_t)B * P), kThreads, 0, F->stream>>>(x, F->half + L.oP, F->master + L.op, F->h, B, C, P);
  const float sc = 1.f / ((float)F->n * (float)F->n);
  for (int l = 0; l < L.layers; ++l) {
    const bool last = l == L.layers - 1;
    float* hin = F->h + (size_t)(keep ? l : (l & 1)) * act_(F);
    float* hout = F->h + (size_t)(keep ? l + 1 : ((l + 1) & 1)) * act_(F);
    launch_analysis(F, hin, B, 1.f, 1.f);
    launch_mix(F, l, F->X + (size_t)l * F->batch * C * modes_(F), B, 0);
    launch_synth_cols(F, B, sc, 2.f * sc);
    SynthArgs a{};
    a.in = hin;
    a.W = F->half + L.oW[l];
    a.bias = F->master + L.ow[l];
    a.act = !last;
    a.out = (last && !keep) ? nullptr : hout;
    a.dact = (keep && !last) ? F->dact + (size_t)l * act_(F) : nullptr;
    if (last) {
      a.Q = F->half + L.oQ;
      a.q = F->master + L.oq;
      a.y = y;
    }
    launch_synth<false>(F, a, B);
  }
  return (int)cudaGetLastError();
}

void weight_gradient(wf_fno_s* F, const float* in, int B, float* gW) {
  const int P = (int)P_(F), C = F->lay.width;
  const int tiles = B * (P / kWgPx), grid = std::min(tiles, 2 * F->sms);
  switch (F->OG) {
    case 1: weight_grad<8><<<grid, 256, wg_smem(8), F->stream>>>(F->gz, in, F->wpart, B, C, P); break;
    case 2: weight_grad<16><<<grid, 256, wg_smem(16), F->stream>>>(F->gz, in, F->wpart, B, C, P); break;
    case 4: weight_grad<32><<<grid, 256, wg_smem(32), F->stream>>>(F->gz, in, F->wpart, B, C, P); break;
    default: weight_grad<64><<<grid, 256, wg_smem(64), F->stream>>>(F->gz, in, F->wpart, B, C, P); break;
  }
  sum_partials<<<(C * C + 31) / 32, 1024, 0, F->stream>>>(F->wpart, grid, C * C, gW, nullptr, 0, C);
}

// loss and gradient of the loss into F->grad (x, t device arrays), after
// forward(..., keep)
int backward(wf_fno_s* F, const float* x, const float* t, int B) {
  const Layout& L = F->lay;
  const int C = L.width, N = F->n, NM = (int)modes_(F), CP = 8 * F->OG;
  const int P = (int)P_(F);
  loss_partial<<<dim3(F->lblk, B), kThreads, 0, F->stream>>>(F->y, t, F->lpart, P);
  loss_fin<<<1, 512, 0, F->stream>>>(F->lpart, F->lblk, B, F->dloss, F->inv);
  // projection Q, and g_z of the last layer
  const float* hL = F->h + (size_t)L.layers * act_(F);
  const int pgrid = std::min(grid_for((size_t)B * P / 4), 4 * F->sms);
  const __half* Q = F->half + L.oQ;
  switch (F->OG) {
    case 1: proj_bwd<8><<<pgrid, kThreads, 0, F->stream>>>(F->y, t, F->inv, Q, hL, F->gz, F->wpart, B, C, P); break;
    case 2: proj_bwd<16><<<pgrid, kThreads, 0, F->stream>>>(F->y, t, F->inv, Q, hL, F->gz, F->wpart, B, C, P); break;
    case 4: proj_bwd<32><<<pgrid, kThreads, 0, F->stream>>>(F->y, t, F->inv, Q, hL, F->gz, F->wpart, B, C, P); break;
    default: proj_bwd<64><<<pgrid, kThreads, 0, F->stream>>>(F->y, t, F->inv, Q, hL, F->gz, F->wpart, B, C, P); break;
  }
  sum_partials<<<(CP + 32) / 32, 1024, 0, F->stream>>>(F->wpart, pgrid, CP + 1, F->grad + L.oQ, F->grad + L.oq, 2, C);
  const float sc = 1.f / ((float)N * (float)N);
  for (int l = L.layers - 1; l >= 0; --l) {
    const float* hin = F->h + (size_t)l * act_(F);
    // spectral branch: g_Y = (c_k / N^2) DFT(g_z), then R and X
    launch_analysis(F, F->gz, B, sc, 2.f * sc);
    launch_mix(F, l, F->gY, B, 1);
    const float2* X = F->X + (size_t)l * F->batch * C * modes_(F);
    mix_bwd_r<<<dim3((NM + 127) / 128, (C + 3) / 4, (C + 3) / 4), 128, 0, F->stream>>>(
        F->gY, X, F->grad + L.oR[l], F->grad + L.ow[l], B, C, NM, (float)N * (float)N);
    launch_synth_cols(F, B, 1.f, 1.f);
    weight_gradient(F, hin, B, F->grad + L.oW[l]);
    // g_h of this layer's input = W^T g_z + Re(inverse of g_X), through the
    // activation below it in place, or into the lift's gradient
    SynthArgs a{};
    a.in = F->gz;
    a.W = F->half + L.oW[l];
    if (l > 0) {
      a.out = F->gz;
      a.mul = F->dact + (size_t)(l - 1) * act_(F);
    } else {
      a.x = x;
      a.lpart = F->wpart;
    }
    const int g = launch_synth<true>(F, a, B);
    if (l == 0)
      sum_partials<<<(CP * 3 + 31) / 32, 1024, 0, F->stream>>>(F->wpart, g, CP * 3, F->grad + L.oP, F->grad + L.op, 1,
                                                              C);
  }
  return (int)cudaGetLastError();
}

int refresh_half(wf_fno_s* F) {
  to_half_kernel<<<grid_for(F->lay.total), kThreads, 0, F->stream>>>(F->master, F->half, F->lay.total);
  return (int)cudaGetLastError();
}

bool dev_ptr(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" {

int wf_fno_create(wf_fno_t* out, int n, int batch, int width, int mx, int my, int layers, const float* params,
                  void* stream) {
  if (!out || !params || n < 16 || n > 1024 || (n & (n - 1)) != 0 || batch < 1 || batch > 64 || width < 1 ||
      width > kMaxWidth || (width & 1) || mx < 1 || mx > kMaxModes || my < 1 || my > kMaxModes || 2 * my > n || mx > n / 2 ||
      layers < 1 || layers > 8)
    return WF_EINVAL;
  wf_fno_s* F = new wf_fno_s();
  F->lay.width = width;
  F->lay.mx = mx;
  F->lay.my = my;
  F->lay.layers = layers;
  F->lay.build();
  F->n = n;
  F->batch = batch;
  F->stream = (cudaStream_t)stream;
  const size_t T = F->lay.total, P = (size_t)n * n;
  F->lblk = 32;
  F->OG = width <= 8 ? 1 : (width <= 16 ? 2 : (width <= 32 ? 4 : 8));
  F->KW = ((mx + 1) / 2 + 7) / 8;  // sets of 8 modes of one parity
  const int CP = 8 * F->OG;
  if (prepare_kernels(F) != cudaSuccess) {
    cudaGetLastError();
    wf_fno_destroy(F);
    return WF_ECUDA;
  }
  // block partial sums: the weight gradients', the projection's, the lift's
  const size_t wpart = std::max((size_t)2 * F->sms * std::max(width * width, 2 * (CP + 1)),
                                (size_t)F->sms * F->adj_per_sm * CP * 3);
  bool ok = alloc(F, &F->master, T) && alloc(F, &F->grad, T) && alloc(F, &F->m1, T) && alloc(F, &F->m2, T) &&
            alloc(F, &F->half, T) && alloc(F, &F->h, (size_t)(layers + 1) * act_(F)) &&
            alloc(F, &F->dact, (size_t)std::max(layers - 1, 1) * act_(F)) && alloc(F, &F->y, (size_t)batch * P) &&
            alloc(F, &F->gz, act_(F)) && alloc(F, &F->Xp, (size_t)batch * width * an_blocks(n) * modes_(F)) &&
            alloc(F, &F->X, (size_t)layers * batch * width * modes_(F)) &&
            alloc(F, &F->gY, (size_t)batch * width * modes_(F)) && alloc(F, &F->Y, (size_t)batch * CP * modes_(F)) &&
            alloc(F, &F->S, (size_t)batch * n * mx * 2 * CP) && alloc(F, &F->tw_x, (size_t)mx * n) &&
            alloc(F, &F->tw_y, (size_t)2 * my * n) && alloc(F, &F->tw_k, (size_t)(n / 2) * 16 * F->KW) &&
            alloc(F, &F->wpart, wpart) && alloc(F, &F->lpart, (size_t)batch * F->lblk * 2) &&
            alloc(F, &F->dloss, 1) && alloc(F, &F->inv, batch);
  if (!ok) {
    wf_fno_destroy(F);
    return WF_ENOMEM;
  }
  // twiddles in double, rounded once
  std::vector<float2> tx((size_t)mx * n), ty((size_t)2 * my * n);
  for (int k = 0; k < mx; ++k)
    for (int x = 0; x < n; ++x) {
      const double a = 2.0 * M_PI * (double)((long long)k * x % n) / n;
      tx[(size_t)k * n + x] = make_float2((float)cos(a), (float)-sin(a));
    }
  for (int j = 0; j < 2 * my; ++j) {
    const int ky = j < my ? j : n - 2 * my + j;
    for (int y = 0; y < n; ++y) {
      const double a = 2.0 * M_PI * (double)((long long)ky * y % n) / n;
      ty[(size_t)j * n + y] = make_float2((float)cos(a), (float)-sin(a));
    }
  }
  // the analysis's row table: [x][parity][k / 2], x < n/2, 0 beyond mx
  std::vector<float2> tk((size_t)(n / 2) * 16 * F->KW, make_float2(0.f, 0.f));
  for (int x = 0; x < n / 2; ++x)
    for (int k = 0; k < mx; ++k) tk[(size_t)x * 16 * F->KW + (k & 1) * 8 * F->KW + k / 2] = tx[(size_t)k * n + x];
  const cudaMemcpyKind k = dev_ptr(params) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  ok = cudaMemcpy(F->tw_x, tx.data(), tx.size() * sizeof(float2), cudaMemcpyHostToDevice) == cudaSuccess &&
       cudaMemcpy(F->tw_y, ty.data(), ty.size() * sizeof(float2), cudaMemcpyHostToDevice) == cudaSuccess &&
       cudaMemcpy(F->tw_k, tk.data(), tk.size() * sizeof(float2), cudaMemcpyHostToDevice) == cudaSuccess &&
       cudaMemcpy(F->master, params, T * sizeof(float), k) == cudaSuccess &&
       cudaMemset(F->m1, 0, T * sizeof(float)) == cudaSuccess && cudaMemset(F->m2, 0, T * sizeof(float)) == cudaSuccess &&
       cudaMemset(F->grad, 0, T * sizeof(float)) == cudaSuccess;
  if (!ok || refresh_half(F) != cudaSuccess || cudaStreamSynchronize(F->stream) != cudaSuccess) {
    cudaGetLastError();
    wf_fno_destroy(F);
    return WF_ECUDA;
  }
  *out = F;
  return WF_OK;
}

void wf_fno_destroy(wf_fno_t F) {
  if (!F) return;
  for (void* p : F->allocs) cudaFree(p);
  delete F;
}

long long wf_fno_num_params(wf_fno_t F) { return F ? (long long)F->lay.total : -1; }

int wf_fno_forward(wf_fno_t F, const float* x, float* y, int nb) {
  if (!F || !x || !y || nb < 1 || nb > F->batch || !dev_ptr(x) || !dev_ptr(y)) return WF_EINVAL;
  if (forward(F, x, y, nb, false)) return WF_ECUDA;
  return cudaStreamSynchronize(F->stream) == cudaSuccess ? WF_OK : WF_ECUDA;
}

int wf_fno_gradient(wf_fno_t F, const float* x, const float* t, int nb, float* grad, double* loss) {
  if (!F || !x || !t || nb < 1 || nb > F->batch || !dev_ptr(x) || !dev_ptr(t)) return WF_EINVAL;
  if (forward(F, x, F->y, nb, true) || backward(F, x, t, nb)) return WF_ECUDA;
  if (grad && cudaMemcpyAsync(grad, F->grad, F->lay.total * sizeof(float), cudaMemcpyDefault, F->stream) != cudaSuccess)
    return WF_ECUDA;
  double l = 0.0;
  if (cudaMemcpyAsync(&l, F->dloss, sizeof(double), cudaMemcpyDeviceToHost, F->stream) != cudaSuccess ||
      cudaStreamSynchronize(F->stream) != cudaSuccess)
    return WF_ECUDA;
  if (loss) *loss = l;
  return WF_OK;
}

int wf_fno_train_step(wf_fno_t F, const float* x, const float* t, int nb, double lr, double* loss) {
  if (!F || !x || !t || nb < 1 || nb > F->batch || !(lr > 0.0) || !dev_ptr(x) || !dev_ptr(t)) return WF_EINVAL;
  if (forward(F, x, F->y, nb, true) || backward(F, x, t, nb)) return WF_ECUDA;
  F->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)F->step), c2 = 1.f - powf(b2, (float)F->step);
  adam_kernel<<<grid_for(F->lay.total), kThreads, 0, F->stream>>>(F->master, F->grad, F->m1, F->m2, F->lay.total,
                                                                  (float)lr, b1, b2, 1e-8f, c1, c2);
  if (refresh_half(F) != cudaSuccess) return WF_ECUDA;
  double l = 0.0;
  if (cudaMemcpyAsync(&l, F->dloss, sizeof(double), cudaMemcpyDeviceToHost, F->stream) != cudaSuccess ||
      cudaStreamSynchronize(F->stream) != cudaSuccess)
    return WF_ECUDA;
  if (loss) *loss = l;
  return WF_OK;
}

int wf_fno_get_params(wf_fno_t F, float* out, int rounded) {
  if (!F || !out) return WF_EINVAL;
  if (!rounded) {
    if (cudaMemcpy(out, F->master, F->lay.total * sizeof(float), cudaMemcpyDefault) != cudaSuccess) return WF_ECUDA;
    return WF_OK;
  }
  // the values the forward pass uses: FP16 matrices, FP32 biases
  std::vector<__half> hh(F->lay.total);
  std::vector<float> mm(F->lay.total);
  if (cudaMemcpy(hh.data(), F->half, F->lay.total * sizeof(__half), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(mm.data(), F->master, F->lay.total * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess)
    return WF_ECUDA;
  std::vector<char> is_bias(F->lay.total, 0);
  for (int o = 0; o < F->lay.width; ++o) is_bias[F->lay.op + o] = 1;
  for (int l = 0; l < F->lay.layers; ++l)
    for (int o = 0; o < F->lay.width; ++o) is_bias[F->lay.ow[l] + o] = 1;
  is_bias[F->lay.oq] = 1;
  for (size_t i = 0; i < F->lay.total; ++i) mm[i] = is_bias[i] ? mm[i] : __half2float(hh[i]);
  return cudaMemcpy(out, mm.data(), F->lay.total * sizeof(float), cudaMemcpyDefault) == cudaSuccess ? WF_OK : WF_ECUDA;
}

int wf_fno_features(int ny, int nx, const float* d, const float* pixel_var, const uint8_t* mask, float* x_out,
                    float* sigma_out, void* stream) {
  if (!d || !pixel_var || !x_out || !sigma_out || ny < 1 || nx < 1) return WF_EINVAL;
  if (!dev_ptr(d) || !dev_ptr(pixel_var) || !dev_ptr(x_out) || !dev_ptr(sigma_out) || (mask && !dev_ptr(mask)))
    return WF_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  const size_t n = (size_t)ny * nx;
  constexpr int nblk = 64;
  double* part = nullptr;
  if (cudaMallocAsync((void**)&part, 2 * nblk * sizeof(double), s) != cudaSuccess) {
    cudaGetLastError();
    return WF_ENOMEM;
  }
  feat_partial<<<nblk, kThreads, 0, s>>>(pixel_var, mask, part, n);
  feat_fin<<<1, 32, 0, s>>>(part, nblk, sigma_out);
  feat_map<<<grid_for(n), kThreads, 0, s>>>(d, pixel_var, mask, sigma_out, x_out, n);
  cudaFreeAsync(part, s);
  return cudaGetLastError() == cudaSuccess ? WF_OK : WF_ECUDA;
}

}  // extern "C"

// Learned inner-solve controller: the MLP 16 -> 64 -> 64 -> 2 (GELU hidden
// layers) that proposes the inner tolerance factor rho_in (in place of Eq.
// inner-tolerance-factor) and the primal weight carried into the next inner
// solve (in place of the restart value of Eq. primal-weight-update).  BF16
// weights, FP32 arithmetic.  Hand-written inference and training kernels:
// forward (with the pre-activations kept for the backward pass), weighted
// squared-error gradient, backward (per-block partial gradients, reduced in
// a fixed order: deterministic), and Adam on FP32 master weights that
// refreshes the BF16 copy.  The network is tiny (5,378 parameters): every block
// keeps its weights in shared memory and works through tiles of samples.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <string>

#include "../../include/pdnqp.h"

namespace pdq {
namespace {

constexpr int kIn = 16, kHid = 64, kOut = 2;
// Parameter layout (row-major, out x in): W1[64][16], b1[64], W2[64][64],
// b2[64], W3[2][64], b3[2].
constexpr int oW1 = 0, oB1 = oW1 + kHid * kIn, oW2 = oB1 + kHid, oB2 = oW2 + kHid * kHid, oW3 = oB2 + kHid,
              oB3 = oW3 + kOut * kHid, kParams = oB3 + kOut;
constexpr int kCache = 2 * kHid;       // z1, z2 per sample
constexpr int kSamplesPerRow = 16;       // the caller's scratch: one row of partial gradients per 16 samples
constexpr int kMaxGradRows = 1 << 16;    // ... so batches up to 1,048,576 samples

static thread_local std::string g_mlp_err;

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
// GELU and its derivative from one erff.
__device__ __forceinline__ float gelu_both(float z, float &deriv) {
  const float e = 1.0f + erff(z * 0.70710678118654752f);
  deriv = 0.5f * e + z * 0.39894228040143268f * expf(-0.5f * z * z);
  return 0.5f * z * e;
}

// Shared-memory row strides (floats): 64 or 16 columns plus 4, so that rows
// taken by neighbouring threads start on different banks.
constexpr int kLd = kHid + 4, kLdX = kIn + 4;
constexpr int kThreads = 128;

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void st4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
// Global rows of the caller: 16-byte accesses when the base allows them.
__device__ __forceinline__ float4 ldg4(const float *p, bool vec) {
  return vec ? ld4(p) : make_float4(p[0], p[1], p[2], p[3]);
}
__device__ __forceinline__ void stg4(float *p, float4 v, bool vec) {
  if (vec) {
    st4(p, v);
  } else {
    p[0] = v.x;
    p[1] = v.y;
    p[2] = v.z;
    p[3] = v.w;
  }
}

// Forward pass as two small GEMMs per tile of S = 16 R samples, FP32 FMA.
// What bounds it: FP32 issue (5,248 FMA and 128 erff a sample).  Thread (tx,
// ty) owns samples ty, ty + 16, ... and hidden units 4 tx .. 4 tx + 3 and 32 +
// those, so an operand read of 16 bytes feeds 16 FMA at R = 8; one warp reads
// 4 sample rows (broadcast to 8 lanes) and one weight row without bank
// conflicts.  Weights stay in shared memory over the tiles of a block.
// Measured on 231,184 samples: see k_mlp_backward.
template <int R>
struct FwdSmem {
  float w1t[kIn * kLd], w2t[kHid * kLd];  // [input][unit], [unit of layer 1][unit of layer 2]
  float b1[kHid], b2[kHid], w3[kOut * kHid], b3[4];
  float X[16 * R * kLdX], H[16 * R * kLd];
};

template <int R>
__global__ void __launch_bounds__(kThreads) k_mlp_forward(const __nv_bfloat16 *wb, const float *x, int B, float *y,
                                                          float *cache, bool vec) {
  constexpr int S = 16 * R;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  FwdSmem<R> &sm = *reinterpret_cast<FwdSmem<R> *>(smem_raw);
  const int t = threadIdx.x, tx = t & 7, ty = t >> 3;
  for (int p = t; p < kHid * kIn; p += kThreads) sm.w1t[(p % kIn) * kLd + p / kIn] = __bfloat162float(wb[oW1 + p]);
  for (int p = t; p < kHid * kHid; p += kThreads) sm.w2t[(p % kHid) * kLd + p / kHid] = __bfloat162float(wb[oW2 + p]);
  if (t < kHid) {
    sm.b1[t] = __bfloat162float(wb[oB1 + t]);
    sm.b2[t] = __bfloat162float(wb[oB2 + t]);
  }
  if (t < kOut * kHid) sm.w3[t] = __bfloat162float(wb[oW3 + t]);
  if (t < kOut) sm.b3[t] = __bfloat162float(wb[oB3 + t]);
  // acc[i][0..3] = units 4 tx .., acc[i][4..7] = units 32 + 4 tx ..
  float acc[R][8];
  auto bias = [&](const float *b) {
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[i][c] = b[(c >> 2) * 32 + 4 * tx + (c & 3)];
  };
  auto gemm = [&](const float *A, int lda, const float *W, int K) {
#pragma unroll 2
    for (int k = 0; k < K; k += 4) {
      float4 a[R];
#pragma unroll
      for (int i = 0; i < R; ++i) a[i] = ld4(A + (i * 16 + ty) * lda + k);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const float4 wl = ld4(W + (k + kk) * kLd + 4 * tx), wh = ld4(W + (k + kk) * kLd + 32 + 4 * tx);
        const float w[8] = {wl.x, wl.y, wl.z, wl.w, wh.x, wh.y, wh.z, wh.w};
#pragma unroll
        for (int i = 0; i < R; ++i) {
          const float v = kk == 0 ? a[i].x : kk == 1 ? a[i].y : kk == 2 ? a[i].z : a[i].w;
#pragma unroll
          for (int c = 0; c < 8; ++c) acc[i][c] = fmaf(w[c], v, acc[i][c]);
        }
      }
    }
  };
  // Pre-activations to the cache, then GELU in place.
  auto activate = [&](long long s0, int off) {
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const long long s = s0 + i * 16 + ty;
      if (cache && s < B) {
        float *c = cache + s * kCache + off + 4 * tx;
        stg4(c, make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]), vec);
        stg4(c + 32, make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]), vec);
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[i][c] = gelu(acc[i][c]);
    }
  };
  const long long tiles = ((long long)B + S - 1) / S;
  for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const long long s0 = tile * S;
    for (int p = t; p < S * kIn; p += kThreads) {
      const long long g = s0 * kIn + p;
      sm.X[(p / kIn) * kLdX + p % kIn] = g < (long long)B * kIn ? x[g] : 0.0f;
    }
    __syncthreads();  // X (and, on the first tile, the weights) written; H of the last tile read
    bias(sm.b1);
    gemm(sm.X, kLdX, sm.w1t, kIn);
    activate(s0, 0);
#pragma unroll
    for (int i = 0; i < R; ++i) {
      float *h = sm.H + (i * 16 + ty) * kLd + 4 * tx;
      st4(h, make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]));
      st4(h + 32, make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]));
    }
    __syncthreads();
    bias(sm.b2);
    gemm(sm.H, kLd, sm.w2t, kHid);
    activate(s0, kHid);
#pragma unroll
    for (int i = 0; i < R; ++i) {
      float o[kOut];
#pragma unroll
      for (int q = 0; q < kOut; ++q) {
        float v = 0.0f;
#pragma unroll
        for (int c = 0; c < 8; ++c) v = fmaf(sm.w3[q * kHid + (c >> 2) * 32 + 4 * tx + (c & 3)], acc[i][c], v);
#pragma unroll
        for (int d = 1; d < 8; d <<= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
        o[q] = v + sm.b3[q];
      }
      const long long s = s0 + i * 16 + ty;
      if (tx < kOut && s < B) y[s * kOut + tx] = tx == 0 ? o[0] : o[1];
    }
  }
}

// Weighted squared error L = sum_s w_s ||y_s - t_s||^2 / sum_s w_s and its
// gradient dL/dy, sums in FP64 and a fixed order.  Thread-local sums of samples
// first + i * step, then the block's sum (thread 0 has it).
__device__ __forceinline__ void wmse_sums(const float *y, const float *t, const float *wt, int B, long long first,
                                          long long step, double &a, double &sw) {
  a = 0.0;
  sw = 0.0;
  for (long long s = first; s < B; s += step) {
    const double ws = wt ? (double)wt[s] : 1.0;
    sw += ws;
    double q = 0.0;
    for (int o = 0; o < kOut; ++o) {
      const double e = (double)y[s * kOut + o] - (double)t[s * kOut + o];
      q += e * e;
    }
    a += ws * q;
  }
}
__device__ __forceinline__ void block_pair_sum(double &a, double &sw) {
  __shared__ double ra[8], rw[8];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    sw += __shfl_xor_sync(0xffffffffu, sw, o);
  }
  if ((threadIdx.x & 31) == 0) {
    ra[threadIdx.x >> 5] = a;
    rw[threadIdx.x >> 5] = sw;
  }
  __syncthreads();
  a = ra[0];
  sw = rw[0];
  for (int k = 1; k < (int)blockDim.x / 32; ++k) {
    a += ra[k];
    sw += rw[k];
  }
  __syncthreads();
}
__device__ __forceinline__ void wmse_grad(const float *y, const float *t, const float *wt, float inv, long long s,
                                          float *dy) {
  const float ws = wt ? wt[s] : 1.0f;
#pragma unroll
  for (int o = 0; o < kOut; ++o) dy[s * kOut + o] = inv * ws * (y[s * kOut + o] - t[s * kOut + o]);
}

// Small batches: one block does both passes.
__global__ void __launch_bounds__(256) k_mlp_wmse(const float *y, const float *t, const float *wt, int B, float *dy,
                                                  float *loss) {
  double a, sw;
  wmse_sums(y, t, wt, B, threadIdx.x, 256, a, sw);
  block_pair_sum(a, sw);
  sw = sw > 0.0 ? sw : 1.0;
  if (threadIdx.x == 0 && loss) *loss = (float)(a / sw);
  const float inv = (float)(2.0 / sw);
  for (long long s = threadIdx.x; s < B; s += 256) wmse_grad(y, t, wt, inv, s, dy);
}

// Large batches: kWmseBlocks blocks form the sums (one block alone is bound by
// its SM's FP64 pipe), which need a place to wait without a workspace of the
// call's own: block b leaves its two sums (four words) in rows 2b and 2b + 1
// of dy.  A second launch reads them in every block and writes the gradient of
// the other rows, a third reads them once more and writes these rows and the
// loss.
constexpr int kWmseBlocks = 152;
constexpr int kWmseHead = 2 * kWmseBlocks;  // rows of dy that hold the sums
constexpr int kWmseOneBlock = 4096;         // batches up to this: one block (two sweeps of 16 samples a thread)

__global__ void __launch_bounds__(256) k_mlp_wmse_sums(const float *y, const float *t, const float *wt, int B,
                                                       float *dy) {
  double a, sw;
  wmse_sums(y, t, wt, B, (long long)blockIdx.x * 256 + threadIdx.x, (long long)kWmseBlocks * 256, a, sw);
  block_pair_sum(a, sw);
  if (threadIdx.x == 0) {
    float *p = dy + 4 * blockIdx.x;
    p[0] = __int_as_float(__double2hiint(a));
    p[1] = __int_as_float(__double2loint(a));
    p[2] = __int_as_float(__double2hiint(sw));
    p[3] = __int_as_float(__double2loint(sw));
  }
}
__device__ __forceinline__ void wmse_total(const float *dy, double &a, double &sw) {
  a = sw = 0.0;
  if (threadIdx.x < kWmseBlocks) {
    const float *p = dy + 4 * threadIdx.x;
    a = __hiloint2double(__float_as_int(p[0]), __float_as_int(p[1]));
    sw = __hiloint2double(__float_as_int(p[2]), __float_as_int(p[3]));
  }
  block_pair_sum(a, sw);
  sw = sw > 0.0 ? sw : 1.0;
}
__global__ void __launch_bounds__(256) k_mlp_wmse_rest(const float *y, const float *t, const float *wt, int B,
                                                       float *dy) {
  double a, sw;
  wmse_total(dy, a, sw);
  const float inv = (float)(2.0 / sw);
  for (long long s = kWmseHead + (long long)blockIdx.x * 256 + threadIdx.x; s < B; s += (long long)gridDim.x * 256)
    wmse_grad(y, t, wt, inv, s, dy);
}
__global__ void __launch_bounds__(256) k_mlp_wmse_head(const float *y, const float *t, const float *wt, float *dy,
                                                       float *loss) {
  double a, sw;
  wmse_total(dy, a, sw);  // ends in a block barrier: every thread has read the sums
  if (threadIdx.x == 0 && loss) *loss = (float)(a / sw);
  const float inv = (float)(2.0 / sw);
  for (int s = threadIdx.x; s < kWmseHead; s += 256) wmse_grad(y, t, wt, inv, s, dy);
}

// Backward pass.  A block takes tiles of S = 8 R samples and keeps the
// gradients of all its tiles in registers (8 x 4 of dW2 and 4 x 2 of dW1 a
// thread), so the partial gradients that k_mlp_grad_reduce sums are one row a
// block instead of one per 16 samples.  Per tile: both activations and their
// derivatives from the cached pre-activations (thread (tx, ty): units 4 tx ..
// 4 tx + 3 of samples ty, ty + 8, ...), dh1 = W2' dz2 and dW2 += dz2 h1' from
// shared memory (10.7 FMA per 16-byte operand read), then dW1 += dz1 x'.  No
// two threads write the same accumulator and every order is fixed:
// deterministic.  What bounds it: FP32 issue and shared-memory reads.
// Measured (GB300, 231,184 samples): a whole step (forward, error, backward,
// Adam) takes 0.349 ms, 19.5 TFLOP/s of FP32; with one sample at a time per
// block of 64 threads (weight reads 32 ways in conflict, 14,449 rows of
// partial gradients, a single-block error) it took 12.76 ms.
template <int R>
struct BwdSmem {
  float w2[kHid * kLd], w3[kOut * kHid];
  float H1[8 * R * kLd], D2[8 * R * kLd], D1[8 * R * kLd], X[8 * R * kLdX];
};

template <int R>
__global__ void __launch_bounds__(kThreads) k_mlp_backward(const __nv_bfloat16 *wb, const float *x, const float *cache,
                                                           const float *dy, int B, float *part, bool vec) {
  constexpr int S = 8 * R;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  BwdSmem<R> &sm = *reinterpret_cast<BwdSmem<R> *>(smem_raw);
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  for (int p = t; p < kHid * kHid; p += kThreads) sm.w2[(p / kHid) * kLd + p % kHid] = __bfloat162float(wb[oW2 + p]);
  if (t < kOut * kHid) sm.w3[t] = __bfloat162float(wb[oW3 + t]);
  __syncthreads();
  const float4 w30 = ld4(sm.w3 + 4 * tx), w31 = ld4(sm.w3 + kHid + 4 * tx);
  float g2[8][4], g1[4][2], gb1[4], gb2[4], g3[kOut][4], gb3[kOut] = {0.0f, 0.0f};
#pragma unroll
  for (int c = 0; c < 4; ++c) {
#pragma unroll
    for (int r = 0; r < 8; ++r) g2[r][c] = 0.0f;
    g1[c][0] = g1[c][1] = gb1[c] = gb2[c] = g3[0][c] = g3[1][c] = 0.0f;
  }
  const long long tiles = ((long long)B + S - 1) / S;
  for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const long long s0 = tile * S;
    float gd1[R][4];  // GELU derivative at z1
    for (int p = t; p < S * kIn; p += kThreads) {
      const long long g = s0 * kIn + p;
      sm.X[(p / kIn) * kLdX + p % kIn] = g < (long long)B * kIn ? x[g] : 0.0f;
    }
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = i * 8 + ty;
      const long long s = s0 + r;
      float z1[4] = {0.f, 0.f, 0.f, 0.f}, z2[4] = {0.f, 0.f, 0.f, 0.f}, dy0 = 0.0f, dy1 = 0.0f;
      if (s < B) {
        const float *c = cache + s * kCache + 4 * tx;
        const float4 a = ldg4(c, vec), b = ldg4(c + kHid, vec);
        z1[0] = a.x, z1[1] = a.y, z1[2] = a.z, z1[3] = a.w;
        z2[0] = b.x, z2[1] = b.y, z2[2] = b.z, z2[3] = b.w;
        dy0 = dy[s * kOut];
        dy1 = dy[s * kOut + 1];
      }
      gb3[0] += dy0;
      gb3[1] += dy1;
      float h1[4], d2[4];
      const float wa[4] = {w30.x, w30.y, w30.z, w30.w}, wc[4] = {w31.x, w31.y, w31.z, w31.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float dv;
        h1[c] = gelu_both(z1[c], gd1[i][c]);
        const float h2 = gelu_both(z2[c], dv);
        g3[0][c] = fmaf(dy0, h2, g3[0][c]);
        g3[1][c] = fmaf(dy1, h2, g3[1][c]);
        d2[c] = fmaf(wc[c], dy1, wa[c] * dy0) * dv;
        gb2[c] += d2[c];
      }
      st4(sm.H1 + r * kLd + 4 * tx, make_float4(h1[0], h1[1], h1[2], h1[3]));
      st4(sm.D2 + r * kLd + 4 * tx, make_float4(d2[0], d2[1], d2[2], d2[3]));
    }
    __syncthreads();
    // dz1 = (W2' dz2) * gelu'(z1) for this thread's samples and units.
    {
      float dh[R][4];
#pragma unroll
      for (int i = 0; i < R; ++i) dh[i][0] = dh[i][1] = dh[i][2] = dh[i][3] = 0.0f;
#pragma unroll 2
      for (int j = 0; j < kHid; j += 4) {
        float4 w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] = ld4(sm.w2 + (j + q) * kLd + 4 * tx);
#pragma unroll
        for (int i = 0; i < R; ++i) {
          const float4 a = ld4(sm.D2 + (i * 8 + ty) * kLd + j);
          const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            dh[i][0] = fmaf(w[q].x, av[q], dh[i][0]);
            dh[i][1] = fmaf(w[q].y, av[q], dh[i][1]);
            dh[i][2] = fmaf(w[q].z, av[q], dh[i][2]);
            dh[i][3] = fmaf(w[q].w, av[q], dh[i][3]);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < R; ++i) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          dh[i][c] *= gd1[i][c];
          gb1[c] += dh[i][c];
        }
        st4(sm.D1 + (i * 8 + ty) * kLd + 4 * tx, make_float4(dh[i][0], dh[i][1], dh[i][2], dh[i][3]));
      }
    }
    // dW2: units 8 ty .. 8 ty + 7 of layer 2, 4 tx .. 4 tx + 3 of layer 1.
#pragma unroll 2
    for (int s = 0; s < S; ++s) {
      const float4 h = ld4(sm.H1 + s * kLd + 4 * tx);
      const float4 a = ld4(sm.D2 + s * kLd + 8 * ty), b = ld4(sm.D2 + s * kLd + 8 * ty + 4);
      const float dv[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        g2[r][0] = fmaf(dv[r], h.x, g2[r][0]);
        g2[r][1] = fmaf(dv[r], h.y, g2[r][1]);
        g2[r][2] = fmaf(dv[r], h.z, g2[r][2]);
        g2[r][3] = fmaf(dv[r], h.w, g2[r][3]);
      }
    }
    __syncthreads();
    // dW1: units 4 tx .. 4 tx + 3, inputs 2 ty and 2 ty + 1.
#pragma unroll 4
    for (int s = 0; s < S; ++s) {
      const float4 d = ld4(sm.D1 + s * kLd + 4 * tx);
      const float x0 = sm.X[s * kLdX + 2 * ty], x1 = sm.X[s * kLdX + 2 * ty + 1];
      const float dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        g1[c][0] = fmaf(dv[c], x0, g1[c][0]);
        g1[c][1] = fmaf(dv[c], x1, g1[c][1]);
      }
    }
    __syncthreads();  // X, H1, D2, D1 read before the next tile overwrites them
  }
  float *out = part + (size_t)blockIdx.x * kParams;
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) out[oW2 + (8 * ty + r) * kHid + 4 * tx + c] = g2[r][c];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    out[oW1 + (4 * tx + c) * kIn + 2 * ty] = g1[c][0];
    out[oW1 + (4 * tx + c) * kIn + 2 * ty + 1] = g1[c][1];
  }
  // Sums over ty (samples of this block split 8 ways) of b1, b2, W3 and b3.
  float *red = sm.H1;  // [8][4][kHid] and 8 x 2 for b3 (S rows of kLd >= 8 * 272: R >= 4; else D2 and D1 follow)
  static_assert(3 * 8 * R * kLd >= 8 * (4 * kHid + 2), "reduction space");
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    float *q = red + ty * 4 * kHid + 4 * tx + c;
    q[0] = gb1[c];
    q[kHid] = gb2[c];
    q[2 * kHid] = g3[0][c];
    q[3 * kHid] = g3[1][c];
  }
  if (tx == 0) {
    red[8 * 4 * kHid + 2 * ty] = gb3[0];
    red[8 * 4 * kHid + 2 * ty + 1] = gb3[1];
  }
  __syncthreads();
  for (int p = t; p < 4 * kHid; p += kThreads) {
    float a = 0.0f;
    for (int k = 0; k < 8; ++k) a += red[k * 4 * kHid + p];
    const int which = p / kHid, j = p % kHid;
    out[which == 0 ? oB1 + j : which == 1 ? oB2 + j : oW3 + (which - 2) * kHid + j] = a;
  }
  if (t < kOut) {
    float a = 0.0f;
    for (int k = 0; k < 8; ++k) a += red[8 * 4 * kHid + 2 * k + t];
    out[oB3 + t] = a;
  }
}

// grad[p] = sum over blocks of part[b][p]: 8 groups of rows b = g, g + 8, ...
// per parameter, then the 8 group sums in order (fixed order).
__global__ void __launch_bounds__(256) k_mlp_grad_reduce(const float *part, int nb, float *grad) {
  __shared__ float red[8][32];
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int p = blockIdx.x * 32 + lane;
  float a = 0.0f;
  if (p < kParams) {
#pragma unroll 8
    for (int b = g; b < nb; b += 8) a += part[(size_t)b * kParams + p];
  }
  red[g][lane] = a;
  __syncthreads();
  if (g == 0 && p < kParams) {
    for (int k = 1; k < 8; ++k) a += red[k][lane];
    grad[p] = a;
  }
}

// Adam (Kingma & Ba) on the FP32 master weights; the BF16 copy is refreshed
// by round-to-nearest-even.
__global__ void k_mlp_adam(float *w, __nv_bfloat16 *wb, const float *g, float *m, float *v, float lr, float b1,
                           float b2, float eps, float c1, float c2) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= kParams) return;
  const float gp = g[p];
  const float mp = b1 * m[p] + (1.0f - b1) * gp;
  const float vp = b2 * v[p] + (1.0f - b2) * gp * gp;
  m[p] = mp;
  v[p] = vp;
  const float wp = w[p] - lr * (mp / c1) / (sqrtf(vp / c2) + eps);
  w[p] = wp;
  wb[p] = __float2bfloat16_rn(wp);
}

__global__ void k_mlp_to_bf16(const float *w, __nv_bfloat16 *wb, int n) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) wb[p] = __float2bfloat16_rn(w[p]);
}

int fail(const char *msg) {
  g_mlp_err = msg;
  return PDNQP_ERR_ARG;
}
int check_launch(const char *what) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    g_mlp_err = std::string(what) + ": " + cudaGetErrorString(e);
    return PDNQP_ERR_CUDA;
  }
  return 0;
}
int rows_for(int B) { return (int)(((long long)B + kSamplesPerRow - 1) / kSamplesPerRow); }
bool overlap(const float *a, size_t na, const float *b, size_t nb) {
  const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
  return x < y + 4 * nb && y < x + 4 * na;
}
bool aligned16(const void *p) { return ((uintptr_t)p & 15) == 0; }

// Tile sizes: the largest whose tiles still give every SM one (152 SMs), so
// that small batches spread over the chip and large ones reuse each weight
// read for 8 samples.
constexpr int kSms = 152;

template <int R>
int launch_forward(const __nv_bfloat16 *wb, const float *x, int B, float *y, float *cache, cudaStream_t s) {
  constexpr int smem = (int)sizeof(FwdSmem<R>);
  if (cudaFuncSetAttribute(k_mlp_forward<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
    return check_launch("k_mlp_forward");
  const long long tiles = ((long long)B + 16 * R - 1) / (16 * R);
  const int nb = (int)(tiles < 3 * kSms ? tiles : 3 * kSms);
  k_mlp_forward<R><<<nb, kThreads, smem, s>>>(wb, x, B, y, cache, aligned16(cache));
  return check_launch("k_mlp_forward");
}

// Blocks (rows of partial gradients written): at most one per tile of 8 R >= 16
// samples, so the rows fit the caller's ceil(batch / 16).
template <int R>
int launch_backward(const __nv_bfloat16 *wb, const float *x, const float *cache, const float *dy, int B, float *scratch,
                    cudaStream_t s, int *nb_out) {
  static_assert(8 * R >= kSamplesPerRow, "more blocks than scratch rows");
  constexpr int smem = (int)sizeof(BwdSmem<R>);
  if (cudaFuncSetAttribute(k_mlp_backward<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
    return check_launch("k_mlp_backward");
  const long long tiles = ((long long)B + 8 * R - 1) / (8 * R);
  const int nb = (int)(tiles < 2 * kSms ? tiles : 2 * kSms);
  k_mlp_backward<R><<<nb, kThreads, smem, s>>>(wb, x, cache, dy, B, scratch, aligned16(cache));
  *nb_out = nb;
  return check_launch("k_mlp_backward");
}

}  // namespace
}  // namespace pdq

extern "C" {

int pdnqp_mlp_param_count(void) { return pdq::kParams; }

int pdnqp_mlp_forward(const uint16_t *w_bf16, const float *x, int batch, float *y, float *cache, void *stream) {
  using namespace pdq;
  if (!w_bf16 || !x || !y || batch < 0) return fail("NULL argument or negative batch");
  if (batch == 0) return 0;
  const __nv_bfloat16 *wb = (const __nv_bfloat16 *)w_bf16;
  cudaStream_t s = (cudaStream_t)stream;
  if (batch >= 128 * kSms) return launch_forward<8>(wb, x, batch, y, cache, s);
  if (batch >= 32 * kSms) return launch_forward<2>(wb, x, batch, y, cache, s);
  return launch_forward<1>(wb, x, batch, y, cache, s);
}

int pdnqp_mlp_wmse(const float *y, const float *target, const float *weight, int batch, float *dy, float *loss,
                   void *stream) {
  using namespace pdq;
  if (!y || !target || !dy || batch < 0) return fail("NULL argument or negative batch");
  if (batch == 0) return 0;
  cudaStream_t s = (cudaStream_t)stream;
  // The head of dy holds sums between the launches: not when dy is one of the inputs.
  const size_t rows = (size_t)batch * kOut;
  const bool in_place = overlap(dy, rows, y, rows) || overlap(dy, rows, target, rows) ||
                        (weight && overlap(dy, rows, weight, (size_t)batch));
  if (batch <= kWmseOneBlock || in_place) {
    k_mlp_wmse<<<1, 256, 0, s>>>(y, target, weight, batch, dy, loss);
  } else {
    k_mlp_wmse_sums<<<kWmseBlocks, 256, 0, s>>>(y, target, weight, batch, dy);
    const long long nb = ((long long)batch - kWmseHead + 255) / 256;
    k_mlp_wmse_rest<<<(int)(nb < 4 * kSms ? nb : 4 * kSms), 256, 0, s>>>(y, target, weight, batch, dy);
    k_mlp_wmse_head<<<1, 256, 0, s>>>(y, target, weight, dy, loss);
  }
  return check_launch("k_mlp_wmse");
}

int pdnqp_mlp_backward(const uint16_t *w_bf16, const float *x, const float *cache, const float *dy, int batch,
                       float *grad, float *scratch, void *stream) {
  using namespace pdq;
  if (!w_bf16 || !x || !cache || !dy || !grad || !scratch || batch < 0) return fail("NULL argument");
  if (rows_for(batch) > kMaxGradRows) return fail("batch too large (at most 65536 x 16 samples)");
  cudaStream_t s = (cudaStream_t)stream;
  if (batch == 0) return cudaMemsetAsync(grad, 0, sizeof(float) * kParams, s) == cudaSuccess ? 0 : PDNQP_ERR_CUDA;
  const __nv_bfloat16 *wb = (const __nv_bfloat16 *)w_bf16;
  int nb = 0;
  const int rc = batch >= 64 * kSms ? launch_backward<8>(wb, x, cache, dy, batch, scratch, s, &nb)
                                    : launch_backward<2>(wb, x, cache, dy, batch, scratch, s, &nb);
  if (rc) return rc;
  k_mlp_grad_reduce<<<(kParams + 31) / 32, 256, 0, s>>>(scratch, nb, grad);
  return check_launch("k_mlp_grad_reduce");
}

int pdnqp_mlp_adam(float *w, uint16_t *w_bf16, const float *grad, float *m, float *v, int step, float lr, float beta1,
                   float beta2, float eps, void *stream) {
  using namespace pdq;
  if (!w || !w_bf16 || !grad || !m || !v || step < 1) return fail("NULL argument or step < 1");
  const float c1 = 1.0f - powf(beta1, (float)step), c2 = 1.0f - powf(beta2, (float)step);
  k_mlp_adam<<<(kParams + 255) / 256, 256, 0, (cudaStream_t)stream>>>(w, (__nv_bfloat16 *)w_bf16, grad, m, v, lr,
                                                                     beta1, beta2, eps, c1, c2);
  return check_launch("k_mlp_adam");
}

int pdnqp_mlp_to_bf16(const float *w, uint16_t *w_bf16, int count, void *stream) {
  using namespace pdq;
  if (!w || !w_bf16 || count < 0) return fail("NULL argument");
  if (count == 0) return 0;
  k_mlp_to_bf16<<<(count + 255) / 256, 256, 0, (cudaStream_t)stream>>>(w, (__nv_bfloat16 *)w_bf16, count);
  return check_launch("k_mlp_to_bf16");
}

const char *pdnqp_mlp_last_error(void) { return pdq::g_mlp_err.c_str(); }

}  // extern "C"

// Kernels of the external KKT test (Sec. 4.1): residuals of Eqs.
// outer-residuals / outer-scales on the original data of Eq. qp, with
// variable-bound violations counted in r_p.  Included by each entry-point
// translation unit (internal linkage).
//
// Every result is a maximum of non-negative numbers, so the blocks join theirs
// in the output itself with integer atomic maxima on the bit patterns (same
// order as the values, and exact in any order): no partial sums, no scratch,
// no reduction launch.  Comparisons on the way use the bit patterns too, which
// keeps them off the narrow FP64 pipe.
#pragma once
#include <cuda_runtime.h>

#include <cmath>

#include "common.cuh"

namespace pdq {
namespace {

__device__ __forceinline__ u64 umax64(u64 a, u64 b) { return a < b ? b : a; }
// |v| as a residual term: +inf when it is not finite.
__device__ __forceinline__ u64 res_bits(double v) { return nonfinite(v) ? kInfBits : abs_bits(v); }
// |v| as a scale term: left out when it is not finite.
__device__ __forceinline__ u64 scale_bits(double v) { return nonfinite(v) ? 0ull : abs_bits(v); }
// |v| with NaN left out (what fmax does with a NaN operand).
__device__ __forceinline__ u64 nonan_bits(double v) { return is_nan_bits(v) ? 0ull : abs_bits(v); }

// A bound of magnitude 1e20 or more on its own side, or NaN (which no value
// compares with), is absent.
__device__ __forceinline__ double lower_bound_of(double v) {
  const u64 b = abs_bits(v);
  return b >= 0x4415af1d78b58c40ull && (__double2hiint(v) < 0 || b > kInfBits) ? -INFINITY : v;  // the bits of 1e20
}
__device__ __forceinline__ double upper_bound_of(double v) {
  const u64 b = abs_bits(v);
  return b >= 0x4415af1d78b58c40ull && (__double2hiint(v) >= 0 || b > kInfBits) ? INFINITY : v;
}
// Distance of v from [lo, hi] as a residual term (0 for NaN: its products show it).
__device__ __forceinline__ u64 violation_bits(double v, double lo, double hi) {
  const long long kv = order_key(v);
  const bool below = kv < order_key(lo), above = kv > order_key(hi) && !below;
  return (below || above) && !is_nan_bits(v) ? res_bits((below ? lo : v) - (below ? v : hi)) : 0ull;
}

// out = {r_p, r_d, s_p, s_d} before the first block joins (the scales are at least 1).
__global__ void k_kkt_init(double *out) {
  if (threadIdx.x < 4) out[threadIdx.x] = threadIdx.x < 2 ? 0.0 : 1.0;
}

struct KktCsr {
  const int *rp, *ci;
  const double *v;
};

// One launch over the column tiles (Q x, A'y: the heavier ones first) and then
// the row tiles (A x), a tile a warp: 32 rows with LONG = false, 8 with true
// (a matrix with long rows).  What bounds it: the FP64 pipe (a multiply-add per
// entry, 22 us at 13 M entries, plus the steps in which the longer rows of a
// tile run alone) and the gathers' latency.  Measured (GB300, whole call):
// 105 us at n = 1e6, m = 5e5, 13 M entries (a thread per row, block partials
// and a final reduction: 317 us), 19.6 us on power-law rows at n = 50,000
// (77 us).
template <bool LONG>
__global__ void __launch_bounds__(kBlock, 3) k_kkt(int n, int m, KktCsr Q, KktCsr At, KktCsr A,
                                                   const double *__restrict__ c, const double *__restrict__ lc,
                                                   const double *__restrict__ uc, const double *__restrict__ lx,
                                                   const double *__restrict__ ux, const double *__restrict__ x,
                                                   const double *__restrict__ y, double *out) {
  constexpr int TR = LONG ? 8 : 32;
  __shared__ Slot<double> slots[LONG ? 1 : kBlock / 32][LONG ? 1 : kTileSlots];
  const int lane = threadIdx.x & 31;
  Slot<double> *buf = slots[LONG ? 0 : threadIdx.x >> 5];
  const long long tn = ((long long)n + TR - 1) / TR, tm = ((long long)m + TR - 1) / TR;
  const long long w0 = ((long long)blockIdx.x * kBlock + threadIdx.x) >> 5, nw = ((long long)gridDim.x * kBlock) >> 5;
  const MulLdg<double> fx{x}, fy{y};
  u64 q[4] = {0ull, 0ull, 0ull, 0ull};  // r_p, r_d, s_p, s_d
  // Entry ranges of this lane's row in a tile (Q and A' or A), loaded a tile ahead.
  int nb[2], ne[2];
  auto ranges = [&](long long w) {
    nb[0] = nb[1] = ne[0] = ne[1] = 0;
    const bool cols = w < tn;
    const long long r = (cols ? w : w - tn) * TR + lane;
    if (lane >= TR || w >= tn + tm || r >= (cols ? n : m)) return;
    const int *rp = cols ? Q.rp : A.rp;
    nb[0] = __ldg(rp + r);
    ne[0] = __ldg(rp + r + 1);
    if (cols && m > 0) {
      nb[1] = __ldg(At.rp + r);
      ne[1] = __ldg(At.rp + r + 1);
    }
  };
  ranges(w0);
  for (long long w = w0; w < tn + tm; w += nw) {
    const int rb[2] = {nb[0], nb[1]}, re[2] = {ne[0], ne[1]};
    ranges(w + nw);
    if (w < tn) {
      const long long i = w * TR + lane;
      const bool ok = lane < TR && i < n;
      double ci = 0.0, lo = 0.0, hi = 0.0, xi = 0.0, sum[2] = {0.0, 0.0};
      if (ok) {
        ci = __ldg(c + i);
        lo = __ldg(lx + i);
        hi = __ldg(ux + i);
        xi = __ldg(x + i);
      }
      if (LONG) {
        sum[0] = tile_long_rows<false, double>(Q.ci, Q.v, rb[0], re[0], fx);
        if (m > 0) sum[1] = tile_long_rows<false, double>(At.ci, At.v, rb[1], re[1], fy);
      } else {
        sum[0] = tile_rows1<false, double>(Q.ci, Q.v, rb[0], re[0], fx, buf);
        if (m > 0) sum[1] = tile_rows1<false, double>(At.ci, At.v, rb[1], re[1], fy, buf);
      }
      if (ok) {
        const double qx = sum[0], aty = sum[1];
        lo = lower_bound_of(lo);
        hi = upper_bound_of(hi);
        q[0] = umax64(q[0], violation_bits(xi, lo, hi));
        double p = xi - (qx + ci + aty);
        if (!is_nan_bits(p)) {
          if (order_key(p) < order_key(lo)) p = lo;
          if (order_key(p) > order_key(hi)) p = hi;
        }
        q[1] = umax64(q[1], res_bits(xi - p));
        q[3] = umax64(q[3], umax64(scale_bits(qx), umax64(nonan_bits(ci), scale_bits(aty))));
      }
    } else {
      const long long j = (w - tn) * TR + lane;
      const bool ok = lane < TR && j < m;
      double lo = 0.0, hi = 0.0;
      if (ok) {
        lo = __ldg(lc + j);
        hi = __ldg(uc + j);
      }
      const double ax = LONG ? tile_long_rows<false, double>(A.ci, A.v, rb[0], re[0], fx)
                             : tile_rows1<false, double>(A.ci, A.v, rb[0], re[0], fx, buf);
      if (ok) {
        lo = lower_bound_of(lo);
        hi = upper_bound_of(hi);
        q[0] = umax64(q[0], violation_bits(ax, lo, hi));
        q[2] = umax64(q[2], umax64(scale_bits(ax), umax64(scale_bits(lo), scale_bits(hi))));
      }
    }
  }
  __shared__ u64 sm[kBlock / 32][4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q[k] = umax64(q[k], __shfl_xor_sync(0xffffffffu, q[k], o));
    if (lane == 0) sm[threadIdx.x >> 5][k] = q[k];
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    u64 a = sm[0][threadIdx.x];
    for (int k = 1; k < kBlock / 32; ++k) a = umax64(a, sm[k][threadIdx.x]);
    // Most blocks find a value at least theirs already there.
    u64 *o = reinterpret_cast<u64 *>(out) + threadIdx.x;
    if (a > *(volatile u64 *)o) atomicMax(o, a);
  }
}

}  // namespace
}  // namespace pdq

// Setup of one inner solve (a0): warm start (Eq. inner-warm-start), penalty and
// inner Ruiz scaling, diagonal steps, the restart metric of the start.  A handful
// of phases over all rows and columns, in one cooperative launch with a grid
// barrier between them (persistent form), or one launch per phase (graph and
// batched forms, which run beside other work).
#pragma once
#include <math.h>

#include "common.cuh"
#include "kernels.cuh"

namespace pdq {
namespace {  // internal linkage: each solver TU owns its kernels

// A vector that entries multiply, and how they are added.
struct AddSquares {
  template <typename Acc>
  __device__ __forceinline__ void operator()(Acc &acc, Acc v, Acc x) const { acc += x * v * v; }
};
template <typename T, typename Add>
struct Against {
  static constexpr int kOrder = 0;
  const T *x;
  __device__ __forceinline__ T gather(int k) const { return x[k]; }
  __device__ __forceinline__ void add(T &acc, T v, T xk) const { Add()(acc, v, xk); }
};

template <typename T>
struct SetupArgs {
  Mat<double> Hd, Ad, Atd;
  const double *c, *z, *lc, *uc, *lx, *ux;
  double *sb, *rb;      // base s and r
  double *xprev, *u;    // the outer iteration's start: x, and (lambda, z) for the Anderson ring (or null)
  double ginv;
  int sweeps;
  T *ex2, *dy2;         // second buffers of the x and row scales (a sweep reads one and writes the other)
  T *qa, *pa;           // sigma d^2 per row, e^2 / m_w per column
};

// The rows or columns of a phase, as in the trial loop: the long ones, one a
// warp, then tiles without them (LONG: tiles of 8).  body(j, valid, rb, re, one)
// for each item; the entry ranges are loaded an item ahead.  flag: dense rows,
// left out (or null).
template <int NM, bool LONG, typename Body>
__device__ __forceinline__ void for_items(GridCtx g, long long nrows, int nlist, const int *list,
                                          const int *const (&rp)[NM], const unsigned char *flag, Body body) {
  constexpr int TR = LONG ? 8 : 32;
  const int lane = threadIdx.x & 31;
  const long long first = (long long)(threadIdx.x >> 5) * g.nb + g.b, step = (long long)(blockDim.x >> 5) * g.nb;
  const long long nlong = LONG ? 0 : nlist, items = nlong + (nrows + TR - 1) / TR;
  long long nj = 0;
  int nb[NM], ne[NM];
  bool nv = false;
  auto fetch = [&](long long i) {
    nv = false;
#pragma unroll
    for (int m = 0; m < NM; ++m) nb[m] = ne[m] = 0;
    if (i >= items) return;
    const bool one = !LONG && i < nlong;
    nj = one ? __ldg(list + i) : (i - nlong) * TR + lane;
    if (!one && (lane >= TR || nj >= nrows)) return;
    if (flag && flag[nj]) return;
    nv = !one || lane == 0;
    bool lng = false;
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      nb[m] = __ldg(rp[m] + nj);
      ne[m] = __ldg(rp[m] + nj + 1);
      lng |= ne[m] - nb[m] > kLongRowEntries;
    }
    if (!LONG && !one && lng) {
      nv = false;
#pragma unroll
      for (int m = 0; m < NM; ++m) ne[m] = nb[m];
    }
  };
  fetch(first);
  for (long long i = first; i < items; i += step) {
    const long long j = nj;
    const bool valid = nv;
    int rb[NM], re[NM];
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      rb[m] = nb[m];
      re[m] = ne[m];
    }
    fetch(i + step);
    body(j, valid, rb, re, !LONG && i < nlong);
  }
}
template <bool LONG, bool IsMax, typename Acc, typename T, typename F>
__device__ __forceinline__ Acc item_sum(bool one, const int *ci, const T *val, int rb, int re, const F &f,
                                        Slot<Acc> *buf) {
  if (LONG) return tile_long_rows<IsMax, Acc>(ci, val, rb, re, f, buf);
  return one ? warp_row<IsMax, Acc>(ci, val, rb, re, f) : tile_rows1<IsMax, Acc, false>(ci, val, rb, re, f, buf);
}
template <bool LONG, bool IsMax, typename Acc, typename T, typename F>
__device__ __forceinline__ void item_pair(bool one, const Mat<T> &A, const Mat<T> &B, const int (&rb)[2],
                                          const int (&re)[2], const F (&f)[2], Slot<Acc> *buf, Acc (&out)[2]) {
  if (LONG || one || sizeof(Acc) == 8) {  // FP64: one after the other, in one warp's buffer of a single matrix
    out[0] = item_sum<LONG, IsMax, Acc>(one, A.ci, A.val, rb[0], re[0], f[0], buf);
    out[1] = item_sum<LONG, IsMax, Acc>(one, B.ci, B.val, rb[1], re[1], f[1], buf);
  } else {
    const int *const ci[2] = {A.ci, B.ci};
    const T *const val[2] = {A.val, B.val};
    tile_rows<2, IsMax, Acc, false>(ci, val, rb, re, f, buf, out);
  }
}

// Dense rows (the split of long_rows_partial): this block's parts of the sum (or
// maximum) over each dense row, and their join for row s by one warp.
template <bool IsMax, typename T, typename F>
__device__ __forceinline__ void dense_parts(const Dev<T> &d, GridCtx g, const F &f) {
  __shared__ double ws[32];
  for (int b = g.b; b < d.lr_nb; b += g.nb) {
    const long long e0 = lr_cut(d.lr_nnz, b, d.lr_nb), e1 = lr_cut(d.lr_nnz, b + 1, d.lr_nb);
    if (e0 >= e1) continue;
    int s = 0;
    while (s + 1 < d.nlr && d.lr_ptr[s + 1] <= e0) ++s;
    for (; s < d.nlr && d.lr_ptr[s] < e1; ++s) {
      const long long a0 = e0 > d.lr_ptr[s] ? e0 : d.lr_ptr[s];
      const long long a1 = e1 < d.lr_ptr[s + 1] ? e1 : d.lr_ptr[s + 1];
      T acc = T(0);
      for (long long k = a0 + threadIdx.x; k < a1; k += blockDim.x) f.add(acc, d.lr_val[k], f.gather(d.lr_ci[k]));
      double v = double(acc);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v = acc_join<IsMax>(v, __shfl_xor_sync(0xffffffffu, v, o));
      if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int w = 1; w < (int)blockDim.x / 32; ++w) v = acc_join<IsMax>(v, ws[w]);
        d.lr_part[(long long)s * kMaxBlocks + b] = v;
      }
      __syncthreads();
    }
  }
}
template <bool IsMax, typename T>
__device__ __forceinline__ double dense_join(const Dev<T> &d, int s) {
  const long long p0 = d.lr_ptr[s], p1 = d.lr_ptr[s + 1], L = d.lr_nnz;
  double a = 0.0;
  for (int b = threadIdx.x & 31; b < d.lr_nb; b += 32) {
    const long long e0 = lr_cut(L, b, d.lr_nb), e1 = lr_cut(L, b + 1, d.lr_nb);
    if (e0 < e1 && e0 < p1 && e1 > p0) a = acc_join<IsMax>(a, __ldcg(d.lr_part + (long long)s * kMaxBlocks + b));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a = acc_join<IsMax>(a, __shfl_xor_sync(0xffffffffu, a, o));
  return a;
}

// Base row j (Eq. inner-warm-start, in FP64) from v = (A x_b)_j: s_b =
// P_[l_c,u_c](v + lambda / sigma) and r_b = v - s_b on inequality rows, r_b = v -
// b_E on equality rows; B w_b, h' = h - B w_b, the base gradients of the s and r
// blocks, the shifted slack bounds, zero corrections, epoch start and averages,
// and the scales before the first sweep (penalty scaling: e_r = 1 / sqrt(sigma)).
template <typename T>
__device__ __forceinline__ void base_row(const Dev<T> &d, const SetupArgs<T> &a, long long j, double v) {
  const double lam = d.lam[j], sig = d.sig[j], yb = d.yb[j], lo = a.lc[j];
  double s = 0.0, r, bw;
  if (j >= d.mE) {
    const double hi = a.uc[j];
    s = clampv<double>(v + lam / sig, lo, hi);
    r = v - s;
    bw = v - s - r;
    d.ls[j] = T(lo - s);
    d.us[j] = T(hi - s);
    d.qs[j] = T(yb);
    d.s[0][j] = T(0);
    d.sst[j] = T(0);
    d.sbar[0][j] = T(0);
    d.es[j] = T(1);
  } else {
    r = v - lo;
    bw = v - r;
  }
  const double h = j < d.mE ? lo : 0.0;
  a.sb[j] = s;
  a.rb[j] = r;
  if (a.u) a.u[j] = lam;
  d.h[j] = T(h);
  d.Bwb[j] = T(bw);
  d.hp[j] = T(h - bw);
  d.qr[j] = T(lam + sig * r + yb);
  d.r[0][j] = T(0);
  d.y[0][j] = T(0);
  d.Bw[0][j] = T(0);
  d.rst[j] = T(0);
  d.yst[j] = T(0);
  d.rbar[0][j] = T(0);
  d.ybar[0][j] = T(0);
  d.sg[j] = T(sig);
  d.er[j] = T(1.0 / sqrt(sig));
  d.dy[j] = T(1);
  a.qa[j] = T(sig);
}

// Order of dense rows (one_row): the FP64 form's; the bulk form's multipliers hold
// FP32 corrections, which do not see it.
template <typename T>
constexpr int kBaseOrder = sizeof(T) == 8 ? 1 : 0;

// Base columns: H x_b and A' y_b in FP64, q'_x = c - z / gamma + H x_b - A' y_b,
// q_x, the shifted bounds, zero corrections with zero cached products.
template <typename T, bool LR, bool RL, bool CL>
__device__ __forceinline__ void setup_base(const Dev<T> &d, const SetupArgs<T> &a, GridCtx g, Slot<double> *buf) {
  const MulLdg<double> fx{d.xb}, fy{d.yb};
  const int *const crp[2] = {a.Hd.rp, a.Atd.rp};
  for_items<2, CL>(g, d.n, d.nlong_c, d.long_c, crp, nullptr,
                   [&](long long i, bool valid, const int(&rb)[2], const int(&re)[2], bool one) {
                     const double hx = item_sum<CL, false, double>(one, a.Hd.ci, a.Hd.val, rb[0], re[0], fx, buf);
                     const double aty = item_sum<CL, false, double>(one, a.Atd.ci, a.Atd.val, rb[1], re[1], fy, buf);
                     if (!valid) return;
                     const double x = d.xb[i], z = a.z[i], q0 = a.c[i] - z * a.ginv;
                     d.qx0[i] = T(q0);
                     d.qx[i] = T(q0 + hx - aty);
                     d.Hxb[i] = T(hx);
                     d.Atyb[i] = T(aty);
                     d.lx[i] = T(a.lx[i] - x);
                     d.ux[i] = T(a.ux[i] - x);
                     d.x[0][i] = T(0);
                     d.Hx[0][i] = T(0);
                     d.Aty[0][i] = T(0);
                     d.xst[i] = T(0);
                     d.xbar[0][i] = T(0);
                     d.Hxbar[0][i] = T(0);
                     d.ex[i] = T(1);
                     a.xprev[i] = x;
                     if (a.u) a.u[d.m + i] = z;
                   });
  if (LR) {  // dense rows: entry by entry (one_row), a warp each, from the last block down
    const int w = (threadIdx.x >> 5) * g.nb + (g.nb - 1 - g.b);
    for (int s = w; s < d.nlr; s += (blockDim.x >> 5) * g.nb) {
      const int j = d.lr_row[s];
      const double v = one_row<false, double>(a.Ad.ci, a.Ad.val, __ldg(a.Ad.rp + j), __ldg(a.Ad.rp + j + 1),
                                              MulLdg<double, kBaseOrder<T>>{d.xb}, buf);
      if ((threadIdx.x & 31) == 0) base_row<T>(d, a, j, v);
    }
  }
  const int *const rrp[1] = {a.Ad.rp};
  for_items<1, RL>(g, d.m, d.nlong_r, d.long_r, rrp, LR ? d.lr_flag : nullptr,
                   [&](long long j, bool valid, const int(&rb)[1], const int(&re)[1], bool one) {
                     double v;
                     if (RL || one) {  // rows above kDenseRow that the split left out keep the order too
                       const MulLdg<double, kBaseOrder<T>> fo{d.xb};
                       v = RL ? tile_long_rows<false, double>(a.Ad.ci, a.Ad.val, rb[0], re[0], fo, buf)
                              : one_row<false, double>(a.Ad.ci, a.Ad.val, __shfl_sync(0xffffffffu, rb[0], 0),
                                                       __shfl_sync(0xffffffffu, re[0], 0), fo, buf);
                     } else {
                       v = item_sum<RL, false, double>(false, a.Ad.ci, a.Ad.val, rb[0], re[0], fx, buf);
                     }
                     if (valid) base_row<T>(d, a, j, v);
                   });
}

// One row's scales after a sweep: l_inf norms of its row of B~ (amax: max_k
// |A_jk e_k|) and of its s and r columns of [[H~, B~^T], [B~, 0]].
template <typename T>
__device__ __forceinline__ void sweep_row(const Dev<T> &d, const SetupArgs<T> &a, const T *dy, T *dyn, long long j,
                                          T amax) {
  const T dj = dy[j], er = d.er[j], sg = d.sg[j];
  T r = fmax(amax * dj, dj * er);
  if (j >= d.mE) {
    const T es = d.es[j], cs = dj * es;
    r = fmax(r, cs);
    if (cs > T(0)) d.es[j] = es * rsqrt_t(cs);
  }
  const T cr = fmax(er * er * sg, dj * er), dn = r > T(0) ? dj * rsqrt_t(r) : dj;
  if (cr > T(0)) d.er[j] = er * rsqrt_t(cr);
  dyn[j] = dn;
  a.qa[j] = sg * dn * dn;
}

// One sweep of the inner Ruiz scaling, old scales in (ex, dy), new ones to (exn,
// dyn): columns max(max_k |e_k H_ki|, max_j |d_j A_ji|) e_i, rows as above.
template <typename T, bool LR, bool RL, bool CL>
__device__ __forceinline__ void setup_sweep(const Dev<T> &d, const SetupArgs<T> &a, const T *ex, T *exn, const T *dy,
                                            T *dyn, GridCtx g, Slot<T> *buf) {
  typedef Against<T, MaxAbs> F;
  if (LR) dense_parts<true>(d, g, F{ex});
  const int *const crp[2] = {d.H.rp, d.At.rp};
  const F f[2] = {{ex}, {dy}};
  for_items<2, CL>(g, d.n, d.nlong_c, d.long_c, crp, nullptr,
                   [&](long long i, bool valid, const int(&rb)[2], const int(&re)[2], bool one) {
                     T v[2];
                     item_pair<CL, true, T>(one, d.H, d.At, rb, re, f, buf, v);
                     if (!valid) return;
                     const T e = ex[i], c = max_abs(v[0], v[1]) * e;
                     exn[i] = c > T(0) ? e * rsqrt_t(c) : e;
                   });
  const int *const rrp[1] = {d.As.rp};
  for_items<1, RL>(g, d.m, d.nlong_r, d.long_r, rrp, LR ? d.lr_flag : nullptr,
                   [&](long long j, bool valid, const int(&rb)[1], const int(&re)[1], bool one) {
                     const T v = item_sum<RL, true, T>(one, d.As.ci, d.As.val, rb[0], re[0], f[0], buf);
                     if (valid) sweep_row<T>(d, a, dy, dyn, j, v);
                   });
}
template <typename T>
__device__ __forceinline__ void setup_sweep_dense(const Dev<T> &d, const SetupArgs<T> &a, const T *dy, T *dyn) {
  for (int s = threadIdx.x >> 5; s < d.nlr; s += blockDim.x >> 5) {
    const T v = T(dense_join<true>(d, s));
    if ((threadIdx.x & 31) == 0) sweep_row<T>(d, a, dy, dyn, d.lr_row[s], v);
  }
}

// Eq. diagonal-scales for the x columns (m_w) and the effective primal step
// tau_eff / (kappa / omega) = e^2 * 0.99 / m_w (Eq. diagonal-steps), and the x
// terms of the start's restart metric (zero corrections).
template <typename T, bool CL>
__device__ __forceinline__ void setup_mw(const Dev<T> &d, const SetupArgs<T> &a, const T *ex, const T *dy, GridCtx g,
                                         Slot<T> *buf, double &q5) {
  const int *const crp[2] = {d.H.rp, d.At.rp};
  const Against<T, AddAbs> f[2] = {{ex}, {dy}};
  const Against<T, AddSquares> f2{a.qa};
  for_items<2, CL>(g, d.n, d.nlong_c, d.long_c, crp, nullptr,
                   [&](long long i, bool valid, const int(&rb)[2], const int(&re)[2], bool one) {
                     T v[2];
                     item_pair<CL, false, T>(one, d.H, d.At, rb, re, f, buf, v);
                     const T b2 = item_sum<CL, false, T>(one, d.At.ci, d.At.val, rb[1], re[1], f2, buf);
                     if (!valid) return;
                     const T e = ex[i], mw = v[0] * e + fmax(v[1] * e, sqrt(b2) * e), imw = T(1) / mw;
                     d.taux[i] = e * e * (T(0.99) / mw);
                     d.itaux[i] = mw / (T(0.99) * e * e);
                     a.pa[i] = e * e * imw;
                     d.ex[i] = e;
                     const double ed = widen(e), qx = widen(d.qx[i]);
                     const double k = clampv<double>(-ed * ed * qx, widen(d.lx[i]), widen(d.ux[i])) * recip(e);
                     q5 += k * k;
                   });
}

// m_w of the s and r columns, their steps, m_y with the dual step eta_eff /
// (kappa omega) = d^2 * 0.99 / m_y, and the row terms of the restart metric.
template <typename T>
__device__ __forceinline__ void my_row(const Dev<T> &d, const T *dy, long long j, T v, double &q4, double &q5) {
  const T dj = dy[j], sg = d.sg[j], er = d.er[j], br = dj * er, mwr = er * er * sg + br;
  d.taur[j] = er * er * (T(0.99) / mwr);
  d.itaur[j] = mwr / (T(0.99) * er * er);
  T my = v * dj * dj + br * br / mwr;
  const double dd = widen(dj), eb = dd * widen(d.hp[j]);
  q4 += eb * eb;
  const double eg = widen(er) * widen(d.qr[j]);
  q5 += eg * eg;
  if (j >= d.mE) {
    const T es = d.es[j], bs = dj * es, mws = fmax(bs, sqrt(sg * bs * bs));
    d.taus[j] = es * es * (T(0.99) / mws);
    d.itaus[j] = mws / (T(0.99) * es * es);
    my += bs * bs / mws;
    const double e = widen(es);
    const double k = clampv<double>(-e * e * widen(d.qs[j]), widen(d.ls[j]), widen(d.us[j])) * recip(es);
    q5 += k * k;
  }
  d.eta[j] = dj * dj * (T(0.99) / my);
  d.ieta[j] = my / (T(0.99) * dj * dj);
  d.dy[j] = dj;
}
template <typename T, bool LR, bool RL>
__device__ __forceinline__ void setup_my(const Dev<T> &d, const SetupArgs<T> &a, const T *dy, GridCtx g, Slot<T> *buf,
                                         double &q4, double &q5) {
  const Against<T, AddSquares> f{a.pa};
  if (LR) dense_parts<false>(d, g, f);
  const int *const rrp[1] = {d.As.rp};
  for_items<1, RL>(g, d.m, d.nlong_r, d.long_r, rrp, LR ? d.lr_flag : nullptr,
                   [&](long long j, bool valid, const int(&rb)[1], const int(&re)[1], bool one) {
                     const T v = item_sum<RL, false, T>(one, d.As.ci, d.As.val, rb[0], re[0], f, buf);
                     if (valid) my_row<T>(d, dy, j, v, q4, q5);
                   });
}

// End of the setup (whole last block): the dense rows, then the restart metric
// of the start and the status from the blocks' sums.
template <typename T, bool LR>
__device__ __forceinline__ void setup_finish(const Dev<T> &d, const T *dy, int nb) {
  __shared__ double extra[2][kTrialThreads / 32];
  double q4 = 0.0, q5 = 0.0;
  if (LR)
    for (int s = threadIdx.x >> 5; s < d.nlr; s += blockDim.x >> 5) {
      const T v = T(dense_join<false>(d, s));
      if ((threadIdx.x & 31) == 0) my_row<T>(d, dy, d.lr_row[s], v, q4, q5);
    }
  if ((threadIdx.x & 31) == 0) {
    extra[0][threadIdx.x >> 5] = q4;
    extra[1][threadIdx.x >> 5] = q5;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const double *part = d.part + P_TRP * kMaxBlocks;
    double a = 0.0, b = 0.0;
    for (int k = threadIdx.x; k < nb; k += 32) {
      a += __ldcg(part + 4 * k);
      b += __ldcg(part + 4 * k + 1);
    }
    a = warp_sum(a);
    b = warp_sum(b);
    if (threadIdx.x == 0) {
      for (int w = 0; w < (int)blockDim.x / 32; ++w) {
        a += extra[0][w];
        b += extra[1][w];
      }
      const double om = d.st->omega;
      d.st->k_restart = sqrt(om * a + b / om);
      d.st->k_last = INFINITY;
      d.st->status = d.st->start_status;
    }
  }
}

template <typename T>
constexpr unsigned setup_smem_bytes() {  // FP64 base products in both forms
  return kTrialThreads / 32 * kTileSlots * (unsigned)sizeof(Slot<double>);
}

// Forms of the launch: a kernel per phase, a cooperative grid, one cluster.
enum : int { kByPhase = 0, kGrid = 1, kCluster = 2 };

// Phases [from, to): 0 base, 1 .. sweeps the Ruiz sweeps, then m_w, then m_y (and
// the end).  In one launch the grid's (cluster's) barrier separates them; a launch
// of a single phase (kByPhase) takes its last block for what the barrier's
// leader does.  What bounds it: at small sizes the barriers (12 phases, about 3 us
// each, where 33 launches took 0.25 ms), at n = 1e6 the gathers of the sweeps.
template <typename T, bool LR, bool RL, bool CL, int FORM>
__global__ void __launch_bounds__(kTrialThreads, 1) k_setup(Dev<T> d, SetupArgs<T> a, int from, int to) {
  constexpr bool COOP = FORM != kByPhase;
  extern __shared__ __align__(16) unsigned char slots[];
  Slot<double> *buf64 = reinterpret_cast<Slot<double> *>(slots) + (threadIdx.x >> 5) * kTileSlots;
  Slot<T> *buf = reinterpret_cast<Slot<T> *>(buf64);
  unsigned *bar = d.ctr + kCtrBar;
  unsigned gen = COOP && threadIdx.x == 0 ? ld_acquire_gpu(bar + kBarGen) : 0u;
  const GridCtx g = hw_grid();
  double q4 = 0.0, q5 = 0.0;
  T *const ex[2] = {d.ex, a.ex2}, *const dy[2] = {d.dy, a.dy2};
  const int S = a.sweeps;
  for (int ph = from; ph < to; ++ph) {
    const int o = ph >= 1 && ph <= S ? (ph - 1) & 1 : S & 1;  // buffer the phase reads
    if (ph == 0) {
      setup_base<T, LR, RL, CL>(d, a, g, buf64);
    } else if (ph <= S) {
      setup_sweep<T, LR, RL, CL>(d, a, ex[o], ex[o ^ 1], dy[o], dy[o ^ 1], g, buf);
    } else if (ph == S + 1) {
      setup_mw<T, CL>(d, a, ex[o], dy[o], g, buf, q5);
    } else {
      setup_my<T, LR, RL>(d, a, dy[o], g, buf, q4, q5);
    }
    // Sums of the last two phases: of both in a cooperative launch, of each in its
    // own slots otherwise (the end adds them).
    const bool sums = ph > S && (!COOP || ph == S + 2);
    if (sums) {
      double v[4] = {q4, q5, 0.0, 0.0};
      block_sums(v, d.part + P_TRP * kMaxBlocks + 4 * (blockIdx.x + (COOP || ph == S + 1 ? 0 : gridDim.x)));
    }
    auto lead = [&] {
      if (LR && ph >= 1 && ph <= S) setup_sweep_dense<T>(d, a, dy[o], dy[o ^ 1]);
      if (ph == S + 2) setup_finish<T, LR>(d, dy[o], COOP ? (int)gridDim.x : 2 * (int)gridDim.x);
      return 0;
    };
    if (COOP) {
      if (((LR && ph >= 1 && ph <= S) || ph == S + 2 ? loop_sync<FORM == kCluster>(bar, gen, lead)
                                                     : loop_sync<FORM == kCluster>(bar, gen)) < 0)
        return;
    } else if ((LR && ph >= 1 && ph <= S) || ph == S + 2) {
      if (arrive_last(d.ctr + 1)) {
        lead();
        if (threadIdx.x == 0) d.ctr[1] = 0u;
      }
    }
  }
}

}  // namespace
}  // namespace pdq

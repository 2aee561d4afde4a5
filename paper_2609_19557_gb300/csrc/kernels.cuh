// CUDA kernels of the PDNQP hot path (Algorithm 4) and of its setup and outer
// glue (Algorithm 3, Sec. 3.1), templated on the storage type T of the inner
// iterates and matrix values (double: plain FP64 form; float: FP32-bulk form).
//
// Coordinates.  The inner iterates live in the outer-scaled, inner-UNSCALED
// coordinates of Eq. inner-qp: w = (x, s_I, r_E, r_I), y, stored as
// corrections from the FP64 base point of the solve (the warm start w_b, y_b):
// w = w_b + dw, y = y_b + dy.  The base enters only through the gradient of
// the inner objective at the base (q' = q + H w_b - B'y_b), the residual
// h' = h - B w_b and the shifted bounds, so the iteration is exactly PDHG on
// (dw, dy) and the FP32-bulk form keeps full relative precision in the
// corrections.  The penalty scaling
// (Eq. inner-penalty-scaling) and the inner Ruiz scaling (Sec. 3.3.2) are the
// diagonal change of variables w = E w~, y = D y~; PDHG in the scaled space is
// exactly PDHG in these coordinates with the effective diagonal steps
// tau_eff = e^2 tau~ and eta_eff = d^2 eta~, and the acceptance test (Eq.
// adaptive-condition) is invariant under it.  So the CSR values of A, A^T and
// Q are never rewritten inside the solve: the scalings only enter the step
// vectors and the scaled restart metric.
//
// H_k = diag(Q + gamma^-1 I, 0, sigma_E, sigma_I) and B = [[A_E, 0, -I, 0],
// [A_I, -I, 0, -I]] are never formed: their s and r blocks are diagonal and
// handled inline, and only the x blocks are SpMVs (Sec. 3.4: one product each
// with Q, A and A^T per trial).
#pragma once
#include <math.h>

#include "common.cuh"

namespace pdq {
namespace {  // internal linkage: each solver TU owns its kernels

// Rows of the partial-sums array used by each reduction.
constexpr int P_TR_R = 0;    // trial, row kernel: lhs_tau, lhs_eta, rhs_h, rhs_b
constexpr int P_TR_C = 4;    // trial, column kernel (same 4)
constexpr int P_CK_R = 8;    // check, row kernel: 16 quantities
constexpr int P_CK_C = 24;   // check, column kernel: 16 quantities
constexpr int P_TRP = 40;    // persistent loop: 4 sums per block, block-major
constexpr unsigned CK_MAXMASK = 0x0F0Fu;  // quantities 0-3 and 8-11 of a check are maxima
// Counter words (d.ctr): [0] column last-block counter, [1] check last-block
// counter, [2] row last-block counter (long rows), [3] outer column last-block counter, [kCtrBar, kCtrBar + kBarWords) the grid barrier of the persistent loop.
constexpr int kCtrBar = 128, kCtrWords = kCtrBar + kBarWords;
// Rows of A with more entries than this are treated as dense coupling rows
// (at most kMaxLong of them, the longest first; the rest stay row-wise).
constexpr int kLongRowMin = kDenseRow;
constexpr int kMaxLong = 64;

template <typename T>
struct Mat {
  int nrows;
  const int *rp;
  const int *ci;
  const T *val;
};

// Device pointers of one solver (passed by value to the trial kernels).
template <typename T>
struct Dev {
  int n, m, mE;
  Mat<T> H, A, At;  // H = Qbar + gamma^-1 I (x block of H_k), A (rows E then I), A^T
  // n-vectors: corrections dx and their cached products H dx, A' dy, averages
  T *x[3], *Hx[2], *Aty[2], *xbar[2], *Hxbar[2];  // x: current, trial and spare (DevState::xcur ..)
  T *qx;          // q'_x = c - z / gamma + H x_b - A' y_b
  T *qx0;         // q_x = c - z / gamma (scale s_d)
  T *Hxb, *Atyb;  // H x_b, A' y_b (scales)
  T *lx, *ux;     // shifted bounds l - x_b, u - x_b
  T *taux, *itaux, *ex, *xst, *Atybar;
  // m-vectors (s is indexed by row; entries of equality rows are unused)
  T *y[2], *s[2], *r[2], *Bw[2], *ybar[2], *sbar[2], *rbar[2];
  T *qs;          // y_b: gradient of the s block at the base (I rows)
  T *qr;          // lambda + sigma r_b + y_b: gradient of the r block at the base
  T *hp;          // h - B w_b
  T *h, *Bwb;     // h and B w_b (scale s_p)
  T *ls, *us;     // shifted slack bounds l_c - s_b, u_c - s_b (I rows)
  T *eta, *taus, *taur, *ieta, *itaus, *itaur, *es, *er, *dy, *yst, *sst, *rst, *Bwbar;
  // FP64 base point and outer data
  const double *xb, *yb, *sb, *rb;  // base: outer x, inner y, warm-start s and r
  const double *lam, *sig;          // multipliers and row penalties
  T *sg;                            // the row penalties in the storage type (constant during an inner solve)
  double *part;
  // Dense coupling rows (more than kLongRowMin entries): their products are
  // split evenly over the blocks of the row pass, and the block that
  // arrives last combines the block partials in block order and updates
  // those rows.  As is A with these rows emptied (As == A when nlr == 0).
  int nlr;
  int lr_nnz;
  int lr_nb;       // parts of the split in the persistent loop
  Mat<T> As;
  const int *lr_row;   // [nlr] row index of each long row (ascending)
  const int *lr_ptr;   // [nlr + 1] offsets into lr_ci / lr_val
  const int *lr_ci;
  const T *lr_val;
  const unsigned char *lr_flag;  // [m] 1 for a long row
  // Rows of As, and variables, with more than kLongRowEntries entries (variables: in H or A'): the persistent loop
  // gives each a warp of its own, so that they do not hold up their tiles.
  int nlong_r, nlong_c;
  const int *long_r, *long_c;
  double *lr_part;     // [kMaxLong][kMaxBlocks] block partial products
  double *lr_acc;      // [4] acceptance-sum terms of the long rows (added to the row sums)
  DevState *st;
  unsigned *ctr;   // arrival counters of the last-block reductions (reset by the last block)
  unsigned long long *ptime;  // persistent loop: ns spent in the primal, row and column(+decision) passes
  cudaGraphConditionalHandle hw, hc;  // device-loop handles (0 when the graph has none)
};

template <typename T>
__device__ __forceinline__ T clampv(T v, T lo, T hi) {
  // Same comparison order as a plain projection: NaN stays NaN.
  v = v < lo ? lo : v;
  v = v > hi ? hi : v;
  return v;
}

// FP64: the same on the integer pipes (a comparison on the FP64 pipe costs as much as a multiply-add).
template <>
__device__ __forceinline__ double clampv<double>(double v, double lo, double hi) {
  const long long k = order_key(v);
  const bool below = k < order_key(lo), above = k > order_key(hi);
  const double p = above ? hi : (below ? lo : v);
  return is_nan_bits(v) ? v : p;
}

#define PDNQP_GRID_STRIDE(i, N) \
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (long long)(N); \
       i += (long long)gridDim.x * blockDim.x)
// The same over the blocks of a GridCtx (one problem's share of a batched launch).
#define PDNQP_VGRID_STRIDE(i, N, g) \
  for (long long i = (long long)(g).b * blockDim.x + threadIdx.x; i < (long long)(N); \
       i += (long long)(g).nb * blockDim.x)

// The single-block kernels work on a shared-memory copy of the device state
// (one coalesced load and store) instead of chains of dependent global
// read-modify-writes.
__device__ __forceinline__ void state_load(DevState &S, const DevState *g) {
  for (int i = threadIdx.x; i < (int)(sizeof(DevState) / 4); i += blockDim.x) ((int *)&S)[i] = __ldcg((const int *)g + i);
  __syncthreads();
}
__device__ __forceinline__ void state_store(DevState *g, const DevState &S) {
  __syncthreads();
  for (int i = threadIdx.x; i < (int)(sizeof(DevState) / 4); i += blockDim.x) ((int *)g)[i] = ((const int *)&S)[i];
}

// Start of one graph launch: at most `chunk` trials before control returns to
// the host.
__global__ void k_loop_begin(DevState *st, long long chunk) { st->slot_left = chunk; }

// Last-block detection: after this block's partial sums are stored, returns
// true in the single block that arrives last (its threads then see every
// block's partials); that block resets the counter at the end of its work.
__device__ __forceinline__ bool arrive_last(unsigned *ctr, int nb = -1) {
  __shared__ bool last;
  if (nb < 0) nb = gridDim.x;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ctr, 1u) == (unsigned)(nb - 1);
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// A kernel that finds the loop stopped ends the device loop (block 0 only).
// COND = false builds kernels without conditional-handle calls (for unrolled
// graphs, which profilers can inspect).
template <bool COND>
__device__ __forceinline__ void stop_loop(cudaGraphConditionalHandle hw, cudaGraphConditionalHandle hc) {
  if (COND && blockIdx.x == 0 && threadIdx.x == 0) {
    if (hw) cudaGraphSetConditional(hw, 0u);
    if (hc) cudaGraphSetConditional(hc, 0u);
  }
}

template <bool COND>
__device__ void decide_body(DevState *stg, const double *part, const double *lacc, int nb_r, int nb_c,
                            cudaGraphConditionalHandle hw, cudaGraphConditionalHandle hc);
template <bool COND>
__device__ void check_final_body(DevState *stg, const double *part, int nb_r, int nb_c,
                                 cudaGraphConditionalHandle hw);
__device__ __forceinline__ bool decide_logic(DevState *st, const double (&a)[4]);
__device__ __forceinline__ void trial_begin(DevState *st);
__device__ __forceinline__ void trial_accept(DevState *st);

// ===========================================================================
// Trial step (Eq. pdqp-trial) and acceptance test (Eq. adaptive-condition).
// ===========================================================================

// Primal x-block of the trial: x_tr = P_[l,u](x - tau (q + (1-alpha) H xbar +
// alpha H x - A'y)) with the cached products H x, H xbar, A'y.
// The phase functions below read the scalar state through `st` (global
// memory in the one-kernel-per-phase launches, a shared-memory copy in the
// persistent loop) and touch the iterate buffers through plain pointers: in
// the persistent loop the same buffers are written and read across grid
// barriers within one launch, so they must not go through the read-only path.
// 16-byte vectors of the streaming passes (every vector is its own
// allocation, so 256-byte aligned): W elements per load or store.
template <typename T>
struct Vec16;
template <>
struct Vec16<float> {
  typedef float4 type;
};
template <>
struct Vec16<double> {
  typedef double2 type;
};
template <typename T>
struct Pack {
  static constexpr int W = 16 / sizeof(T);
  T v[W];
  __device__ __forceinline__ void load(const T *p, long long i) {
    *reinterpret_cast<typename Vec16<T>::type *>(v) = reinterpret_cast<const typename Vec16<T>::type *>(p)[i];
  }
  __device__ __forceinline__ void store(T *p, long long i) const {
    reinterpret_cast<typename Vec16<T>::type *>(p)[i] = *reinterpret_cast<const typename Vec16<T>::type *>(v);
  }
};

template <typename T>
__device__ __forceinline__ void primal_phase(const Dev<T> &d, const DevState *st, GridCtx g = hw_grid()) {
  const int cur = st->cur, a0 = st->acur, acc = st->accepted;
  const Scal<T> k0(st);
  const T alpha = k0[kAlpha], oma = k0[kOma], sc = k0[kSct], ap = k0[kAp], omap = k0[kOmap];
  const T *x = d.x[st->xcur];
  const T *Hx = d.Hx[cur];
  const T *Aty = d.Aty[cur];
  T *xt = d.x[st->xtr];
  constexpr int W = Pack<T>::W;
  const long long nv = d.n / W;
  // W elements per thread and trip with 16-byte loads and stores; the same
  // arithmetic per element as the scalar tail below.
  PDNQP_VGRID_STRIDE(c, nv, g) {
    Pack<T> X, HX, HB, Q, AT, TA, L, U, XT;
    X.load(x, c);
    HX.load(Hx, c);
    HB.load(d.Hxbar[a0], c);
    Q.load(d.qx, c);
    AT.load(Aty, c);
    TA.load(d.taux, c);
    L.load(d.lx, c);
    U.load(d.ux, c);
    if (acc) {
      // Running averages of the previous acceptance (Algorithm 4), written to
      // the other buffer: wbar <- (1 - alpha) wbar + alpha w.
      Pack<T> XB;
      XB.load(d.xbar[a0], c);
#pragma unroll
      for (int k = 0; k < W; ++k) {
        HB.v[k] = omap * HB.v[k] + ap * HX.v[k];
        XB.v[k] = omap * XB.v[k] + ap * X.v[k];
      }
      HB.store(d.Hxbar[a0 ^ 1], c);
      XB.store(d.xbar[a0 ^ 1], c);
    }
#pragma unroll
    for (int k = 0; k < W; ++k) {
      const T g = Q.v[k] + oma * HB.v[k] + alpha * HX.v[k] - AT.v[k];
      XT.v[k] = clampv<T>(X.v[k] - (sc * TA.v[k]) * g, L.v[k], U.v[k]);
    }
    XT.store(xt, c);
  }
  // Tail (n mod W elements).
  const long long tid = (long long)g.b * blockDim.x + threadIdx.x;
  const long long i = nv * W + tid;
  if (i < d.n) {
    const T xi = x[i], hxi = Hx[i];
    T hxb;
    if (acc) {
      hxb = omap * d.Hxbar[a0][i] + ap * hxi;
      d.Hxbar[a0 ^ 1][i] = hxb;
      d.xbar[a0 ^ 1][i] = omap * d.xbar[a0][i] + ap * xi;
    } else {
      hxb = d.Hxbar[a0][i];
    }
    const T g = d.qx[i] + oma * hxb + alpha * hxi - Aty[i];
    xt[i] = clampv<T>(xi - (sc * d.taux[i]) * g, d.lx[i], d.ux[i]);
  }
}

template <typename T>
__global__ void __launch_bounds__(kBlock) k_primal(Dev<T> d) {
  if (d.st->status != ST_RUNNING) return;
  primal_phase<T>(d, d.st);
}

// ---------------------------------------------------------------------------
// Dense coupling rows.  Block b of the row pass forms the products of entries
// [b L / nb, (b + 1) L / nb) of the concatenated long rows (L entries in all)
// and stores one partial per long row it touches (FP64, block order fixed);
// the block that arrives last sums, for each long row, the partials of the
// blocks whose range overlaps it, in block order, and applies the row update
// of the trial to those rows.  Deterministic for a given grid size.
// ---------------------------------------------------------------------------
__device__ __forceinline__ long long lr_cut(long long L, int b, int nb) { return L * b / nb; }

// Sum of one double per thread, in a fixed order; the result is in thread 0.
__device__ __forceinline__ double block_sum_fixed(double v) {
  __shared__ double ws[32];
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
  __syncthreads();
  double a = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)blockDim.x / 32; ++w) a += ws[w];
  __syncthreads();
  return a;
}

template <typename T>
__device__ __forceinline__ void long_rows_partial(const Dev<T> &d, const T *xt, GridCtx g = hw_grid()) {
  const long long L = d.lr_nnz;
  const int nb = g.nb, b = g.b;
  const long long e0 = lr_cut(L, b, nb), e1 = lr_cut(L, b + 1, nb);
  if (e0 >= e1) return;
  int s = 0;
  while (s + 1 < d.nlr && d.lr_ptr[s + 1] <= e0) ++s;
  for (; s < d.nlr && d.lr_ptr[s] < e1; ++s) {
    const long long a0 = e0 > d.lr_ptr[s] ? e0 : d.lr_ptr[s];
    const long long a1 = e1 < d.lr_ptr[s + 1] ? e1 : d.lr_ptr[s + 1];
    T acc = T(0);
    if (threadIdx.x < kBlock)
      for (long long k = a0 + threadIdx.x; k < a1; k += kBlock) acc += d.lr_val[k] * __ldcg(xt + d.lr_ci[k]);
    const double v = block_sum_fixed(double(acc));
    if (threadIdx.x == 0) d.lr_part[(long long)s * kMaxBlocks + b] = v;
  }
}

// Row update of one constraint row with (A x_tr)_j = ax: the same arithmetic
// as the row passes below (one thread).
template <typename T>
__device__ __forceinline__ void row_update_one(const Dev<T> &d, const DevState *st, long long j, T ax, T &Lt, T &Le,
                                               T &RH, T &RB) {
  const int cur = st->cur, nx = 1 - cur, a0 = st->acur, acc = st->accepted;
  const Scal<T> k0(st);
  const T alpha = k0[kAlpha], oma = k0[kOma], beta = k0[kBeta], sct = k0[kSct], sce = k0[kSce], ap = k0[kAp],
          omap = k0[kOmap];
  const bool ineq = j >= d.mE;
  const T y = d.y[cur][j], r = d.r[cur][j];
  T rb;
  if (acc) {
    rb = omap * d.rbar[a0][j] + ap * r;
    d.rbar[a0 ^ 1][j] = rb;
    d.ybar[a0 ^ 1][j] = omap * d.ybar[a0][j] + ap * y;
    if (ineq) d.sbar[a0 ^ 1][j] = omap * d.sbar[a0][j] + ap * d.s[cur][j];
  } else {
    rb = d.rbar[a0][j];
  }
  const T sig = T(d.sig[j]);
  const T rt = r - (sct * d.taur[j]) * (d.qr[j] + sig * (oma * rb + alpha * r) + y);
  d.r[nx][j] = rt;
  T bwt = ax - rt, ds = T(0);
  if (ineq) {
    const T s0 = d.s[cur][j];
    const T stv = clampv<T>(s0 - (sct * d.taus[j]) * (d.qs[j] + y), d.ls[j], d.us[j]);
    d.s[nx][j] = stv;
    ds = stv - s0;
    Lt += ds * ds * d.itaus[j];
    bwt -= stv;
  }
  const T yt = y + (sce * d.eta[j]) * (d.hp[j] - bwt - beta * (bwt - d.Bw[cur][j]));
  d.Bw[nx][j] = bwt;
  d.y[nx][j] = yt;
  const T dr = rt - r, dyv = yt - y;
  Lt += dr * dr * d.itaur[j];
  Le += dyv * dyv * d.ieta[j];
  RH += fabs(dr * sig * dr);
  RB += fabs(ds * dyv) + fabs(dr * dyv);
}

// Run by one whole block once every block's partials are visible (nb = the
// row pass's grid size).  The warps take the long rows in turn; the four
// acceptance-sum terms go to lr_acc (warps combined in order).
template <typename T>
__device__ void long_rows_finish(const Dev<T> &d, const DevState *st, int nb) {
  __shared__ double wacc[32][4];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const long long L = d.lr_nnz;
  T Lt = T(0), Le = T(0), RH = T(0), RB = T(0);
  for (int s = w; s < d.nlr; s += nw) {
    const long long p0 = d.lr_ptr[s], p1 = d.lr_ptr[s + 1];
    double a = 0.0;
    for (int b = lane; b < nb; b += 32) {
      const long long e0 = lr_cut(L, b, nb), e1 = lr_cut(L, b + 1, nb);
      if (e0 < e1 && e0 < p1 && e1 > p0) a += __ldcg(d.lr_part + (long long)s * kMaxBlocks + b);
    }
    a = warp_sum(a);
    if (lane == 0) row_update_one<T>(d, st, d.lr_row[s], T(a), Lt, Le, RH, RB);
  }
  if (lane == 0) {
    wacc[w][0] = double(Lt);
    wacc[w][1] = double(Le);
    wacc[w][2] = double(RH);
    wacc[w][3] = double(RB);
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double v = 0.0;
    for (int k = 0; k < nw; ++k) v += wacc[k][threadIdx.x];
    d.lr_acc[threadIdx.x] = v;
  }
  __syncthreads();
}

// Constraint rows: (A x_tr)_j, the s/r blocks of the primal trial, B w_tr,
// the dual trial y_tr = y + eta (h - B w_tr - beta (B w_tr - B w)), and the
// row-local terms of the acceptance sums.  Steps are used as
// tau = (kappa / omega) tau0, eta = (kappa omega) eta0; the sums of
// dw^2 / tau and dy^2 / eta are accumulated with the stored inverses 1/tau0,
// 1/eta0 and scaled once by omega / kappa and 1 / (kappa omega).
template <typename T, int G>
__device__ __forceinline__ void rows_phase(const Dev<T> &d, const DevState *st, GridCtx g = hw_grid()) {
  const int cur = st->cur, nx = 1 - cur, a0 = st->acur, acc = st->accepted;
  const Scal<T> k0(st);
  const T alpha = k0[kAlpha], oma = k0[kOma], beta = k0[kBeta], sct = k0[kSct], sce = k0[kSce], ap = k0[kAp],
          omap = k0[kOmap];
  const T *xt = d.x[st->xtr];
  T Lt = T(0), Le = T(0), RH = T(0), RB = T(0);
  TileIter<G> ti(g);
  for (long long tile = ti.first; tile < d.m; tile += ti.step) {
    long long j;
    const bool own = ti.row(tile, d.m, j);
    const bool valid = own && !(d.nlr && d.lr_flag[j]), ineq = j >= d.mE;
    // Everything that does not need (A x_tr)_j first (the r and s blocks of
    // the trial and the operands of the dual step), so that these loads
    // overlap the SpMV chain.
    T y = T(0), r = T(0), rt = T(0), stv = T(0), ds = T(0), bw = T(0), etj = T(0), hpj = T(0), sig = T(0);
    if (valid) {
      y = d.y[cur][j];
      r = d.r[cur][j];
      T rb;
      if (acc) {  // running averages of the previous acceptance
        rb = omap * d.rbar[a0][j] + ap * r;
        d.rbar[a0 ^ 1][j] = rb;
        d.ybar[a0 ^ 1][j] = omap * d.ybar[a0][j] + ap * y;
        if (ineq) d.sbar[a0 ^ 1][j] = omap * d.sbar[a0][j] + ap * d.s[cur][j];
      } else {
        rb = d.rbar[a0][j];
      }
      sig = T(d.sig[j]);
      rt = r - (sct * d.taur[j]) * (d.qr[j] + sig * (oma * rb + alpha * r) + y);
      d.r[nx][j] = rt;
      if (ineq) {
        const T s = d.s[cur][j];
        stv = clampv<T>(s - (sct * d.taus[j]) * (d.qs[j] + y), d.ls[j], d.us[j]);
        d.s[nx][j] = stv;
        ds = stv - s;
        Lt += ds * ds * d.itaus[j];
      }
      bw = d.Bw[cur][j];
      etj = d.eta[j];
      hpj = d.hp[j];
    }
    const T ax = tile_row_sum<G, T>(d.As.rp, d.As.ci, d.As.val, tile, d.m, MulLd<T>{xt});
    if (valid) {
      T bwt = ax - rt;
      if (ineq) bwt -= stv;
      const T yt = y + (sce * etj) * (hpj - bwt - beta * (bwt - bw));
      d.Bw[nx][j] = bwt;
      d.y[nx][j] = yt;
      const T dr = rt - r, dyv = yt - y;
      Lt += dr * dr * d.itaur[j];
      Le += dyv * dyv * d.ieta[j];
      RH += fabs(dr * sig * dr);
      RB += fabs(ds * dyv) + fabs(dr * dyv);
    }
  }
  double v[4] = {double(Lt), double(Le), double(RH), double(RB)};
  block_reduce_store<4, 0u>(v, d.part + P_TR_R * kMaxBlocks, g.b);
}

// Row pass of one trial over the blocks of g (graph and batched forms).
template <typename T, int G>
__device__ __forceinline__ void rows_trial_body(const Dev<T> &d, GridCtx g) {
  if (d.st->status != ST_RUNNING || d.st->check_due) return;
  if (d.nlr) long_rows_partial<T>(d, d.x[d.st->xtr], g);
  rows_phase<T, G>(d, d.st, g);
  if (d.nlr && arrive_last(d.ctr + 2, g.nb)) {
    long_rows_finish<T>(d, d.st, g.nb);
    if (threadIdx.x == 0) d.ctr[2] = 0u;
  }
}

template <typename T, int G>
__global__ void __launch_bounds__(kBlock) k_rows(Dev<T> d) {
  rows_trial_body<T, G>(d, hw_grid());
}

// Variable rows: (H x_tr)_i and (A' y_tr)_i (the products with Q and A^T),
// plus the x terms of the acceptance sums.
template <typename T, int G>
__device__ __forceinline__ void cols_phase(const Dev<T> &d, const DevState *st, GridCtx g = hw_grid()) {
  const int cur = st->cur, nx = 1 - cur;
  const T *xt = d.x[st->xtr], *xc = d.x[st->xcur];
  const T *yt = d.y[nx];
  T Lt = T(0), RH = T(0), RB = T(0);
  TileIter<G> ti(g);
  for (long long tile = ti.first; tile < d.n; tile += ti.step) {
    long long i;
    const bool own = ti.row(tile, d.n, i);
    // Row-local operands first: their loads overlap the SpMV chains.
    T xti = T(0), xci = T(0), hxc = T(0), atc = T(0), itx = T(0);
    if (own) {
      xti = xt[i];
      xci = xc[i];
      hxc = d.Hx[cur][i];
      atc = d.Aty[cur][i];
      itx = d.itaux[i];
    }
    const T hx = tile_row_sum<G, T>(d.H.rp, d.H.ci, d.H.val, tile, d.n, MulLd<T>{xt});
    const T aty = tile_row_sum<G, T>(d.At.rp, d.At.ci, d.At.val, tile, d.n, MulLd<T>{yt});
    if (own) {
      d.Hx[nx][i] = hx;
      d.Aty[nx][i] = aty;
      const T dx = xti - xci;
      const T dh = hx - hxc;
      const T da = aty - atc;
      Lt += dx * dx * itx;
      RH += fabs(dx * dh);
      RB += fabs(dx * da);
    }
  }
  double v[4] = {double(Lt), 0.0, double(RH), double(RB)};
  block_reduce_store<4, 0u>(v, d.part + P_TR_C * kMaxBlocks, g.b);
}

// Column pass of one trial over the blocks of g, with the acceptance decision
// in the problem's last block (graph and batched forms).
template <typename T, int G, bool COND>
__device__ __forceinline__ void cols_trial_body(const Dev<T> &d, int nb_r, GridCtx g) {
  if (d.st->status != ST_RUNNING || d.st->check_due) {
    stop_loop<COND>(d.hw, d.hc);
    return;
  }
  cols_phase<T, G>(d, d.st, g);
  if (arrive_last(d.ctr, g.nb)) {
    decide_body<COND>(d.st, d.part, d.nlr ? d.lr_acc : nullptr, nb_r, g.nb, d.hw, d.hc);
    if (threadIdx.x == 0) d.ctr[0] = 0u;
  }
}

template <typename T, int G, bool COND>
__global__ void __launch_bounds__(kBlock) k_cols(Dev<T> d, int nb_r) {
  cols_trial_body<T, G, COND>(d, nb_r, hw_grid());
}

// ===========================================================================
// Persistent trial loop.  One block per SM (fewer for small problems), whose
// warps take tiles of consecutive rows (columns) and work independently: per
// tile the row-local operands, the entries and the gathers are all in flight
// before the first is used, and the arithmetic and the stores follow.
// ===========================================================================
// Threads of a block: 16 warps with 128 registers a thread hold the 16 gathers
// and 11 row-local operands of a column tile without spills where rows are short
// (the FP64 forms of tiles of 8 long rows spill 96 to 184 bytes), and saturate the
// gathers (an SM takes about one 32-byte sector a cycle at random addresses,
// measured with 16 to 64 warps); one block per SM makes the grid barrier and
// the final reduction of the acceptance sums cheap.
constexpr int kTrialThreads = 512;
// Slots of tile_rows (FP64).
template <typename T>
constexpr unsigned trials_smem_bytes() {
  return sizeof(T) == 4 ? 0u : kTrialThreads / 32 * kTileSlots * (unsigned)sizeof(Slot<T>);
}

// The work items of this warp: item w gridDim + b first, so that the last,
// partial round of a pass is spread over all SMs.
struct WarpItems {
  long long first, step;
  int lane;
  __device__ __forceinline__ WarpItems() {
    lane = threadIdx.x & 31;
    first = (long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    step = (long long)(blockDim.x >> 5) * gridDim.x;
  }
};

// This thread's terms of the acceptance sums of a trial, over its rows and
// columns: dw^2 / tau0, dy^2 / eta0, |dw'H dw|, |dw'B'dy|.
template <typename T>
struct TrialSums {
  T Lt, Le, RH, RB;
};

// Row pass: (A x_tr)_j, the s and r blocks of the primal trial, the dual trial
// and the averages of the previous acceptance (the arithmetic of rows_phase).
// Items: the rows of more than kLongRowEntries entries, one a warp, then the
// tiles of 32 rows without them (LONG: tiles of 8 rows, whatever their length).
template <typename T, bool LR, bool LONG>
__device__ __forceinline__ void rows_phase_tiles(const Dev<T> &d, const DevState *st, Slot<T> *buf, TrialSums<T> &ts) {
  constexpr int TR = LONG ? 8 : 32;
  const int cur = st->cur, nx = 1 - cur, a0 = st->acur, acc = st->accepted;
  const Scal<T> k0(st);
  const T *xt = d.x[st->xtr];
  // The split of the dense rows is the instance's own (lr_nb parts), whatever the grid.
  if (LR)
    for (int b = blockIdx.x; b < d.lr_nb; b += gridDim.x) long_rows_partial<T>(d, xt, GridCtx{b, d.lr_nb});
  const WarpItems it;
  const long long nlong = LONG ? 0 : d.nlong_r, items = nlong + ((long long)d.m + TR - 1) / TR;
  const int *ci = d.As.ci;
  const T *val = d.As.val;
  const MulLd<T> f{xt};
  // Row of this lane in an item and its entry range, an item ahead.
  long long nj = 0;
  int nb = 0, ne = 0;
  bool nv = false;
  auto fetch = [&](long long i) {
    nv = false;
    nb = ne = 0;
    if (i >= items) return;
    if (!LONG && i < nlong) {
      nj = __ldg(d.long_r + i);
      nv = it.lane == 0;
      nb = __ldg(d.As.rp + nj);
      ne = __ldg(d.As.rp + nj + 1);
      return;
    }
    nj = (i - nlong) * TR + it.lane;
    if (it.lane >= TR || nj >= d.m) return;
    nb = __ldg(d.As.rp + nj);
    ne = __ldg(d.As.rp + nj + 1);
    nv = !(LR && d.lr_flag[nj]);
    if (!LONG && ne - nb > kLongRowEntries) {
      nv = false;
      ne = nb;
    }
  };
  fetch(it.first);
  for (long long i = it.first; i < items; i += it.step) {
    const long long j = nj;
    const int rb = nb, re = ne;
    const bool valid = nv, ineq = valid && j >= d.mE;
    T y = T(0), r = T(0), rbar = T(0), yb = T(0), tr = T(0), qr = T(0), bw = T(0), eta = T(0), hp = T(0), itr = T(0),
      ie = T(0), sig = T(0), s = T(0), sb = T(0), tus = T(0), qs = T(0), ls = T(0), us = T(0), its = T(0);
    if (valid) {
      y = d.y[cur][j];
      r = d.r[cur][j];
      rbar = d.rbar[a0][j];
      if (acc) yb = d.ybar[a0][j];
      sig = d.sg[j];
      tr = d.taur[j];
      qr = d.qr[j];
      bw = d.Bw[cur][j];
      eta = d.eta[j];
      hp = d.hp[j];
      itr = d.itaur[j];
      ie = d.ieta[j];
    }
    if (ineq) {
      s = d.s[cur][j];
      if (acc) sb = d.sbar[a0][j];
      tus = d.taus[j];
      qs = d.qs[j];
      ls = d.ls[j];
      us = d.us[j];
      its = d.itaus[j];
    }
    fetch(i + it.step);
    T ax;
    if (LONG)
      ax = tile_long_rows<false, T>(ci, val, rb, re, f);
    else if (i < nlong)
      ax = warp_row<false, T>(ci, val, rb, re, f);
    else
      ax = tile_rows1<false, T, false>(ci, val, rb, re, f, buf);
    if (valid) {
      if (acc) {  // running averages of the previous acceptance
        rbar = k0[kOmap] * rbar + k0[kAp] * r;
        d.rbar[a0 ^ 1][j] = rbar;
        d.ybar[a0 ^ 1][j] = k0[kOmap] * yb + k0[kAp] * y;
        if (ineq) d.sbar[a0 ^ 1][j] = k0[kOmap] * sb + k0[kAp] * s;
      }
      const T rt = r - (k0[kSct] * tr) * (qr + sig * (k0[kOma] * rbar + k0[kAlpha] * r) + y);
      d.r[nx][j] = rt;
      T bwt = ax - rt, ds = T(0);
      if (ineq) {
        const T stv = clampv<T>(s - (k0[kSct] * tus) * (qs + y), ls, us);
        d.s[nx][j] = stv;
        ds = stv - s;
        ts.Lt += ds * ds * its;
        bwt -= stv;
      }
      const T yt = y + (k0[kSce] * eta) * (hp - bwt - k0[kBeta] * (bwt - bw));
      d.Bw[nx][j] = bwt;
      d.y[nx][j] = yt;
      const T dr = rt - r, dyv = yt - y, dr2 = dr * dr;
      ts.Lt += dr2 * itr;
      ts.Le += dyv * dyv * ie;
      ts.RH += dr2 * sig;
      ts.RB += fabs(dyv) * (fabs(ds) + fabs(dr));
    }
  }
}

// Column pass: H x_tr and A' y_tr, the
// per-variable terms of the acceptance sums, and, as if the trial were
// accepted, the averages of x and H x and the primal step of the next trial
// (primal_phase with t advanced by one) into the other average buffers and the
// spare x buffer: an acceptance, nearly every trial, then goes on with the row
// pass, without the primal pass (which would read 9 vectors again), its barrier
// and its latency.  A rejection finds the buffers it goes on from untouched.
template <typename T, bool LONG>
__device__ __forceinline__ void cols_phase_tiles(const Dev<T> &d, const DevState *st, Slot<T> *buf, TrialSums<T> &ts) {
  constexpr int TR = LONG ? 8 : 32;
  const int cur = st->cur, nx = 1 - cur, a1 = st->acur ^ st->accepted;  // committed by this trial's passes
  const Scal<T> k0(st);
  const WarpItems it;
  const long long nlong = LONG ? 0 : d.nlong_c, items = nlong + ((long long)d.n + TR - 1) / TR;
  const int *const ci[2] = {d.H.ci, d.At.ci};
  const T *const val[2] = {d.H.val, d.At.val};
  const T *xt = d.x[st->xtr], *xc = d.x[st->xcur];
  T *xs = d.x[st->xsp];
  const MulLd<T> f[2] = {{xt}, {d.y[nx]}};
  long long nj = 0;
  int nb[2] = {0, 0}, ne[2] = {0, 0};
  bool nv = false;
  auto fetch = [&](long long i) {
    nv = false;
    nb[0] = ne[0] = nb[1] = ne[1] = 0;
    if (i >= items) return;
    const bool one = !LONG && i < nlong;
    nj = one ? __ldg(d.long_c + i) : (i - nlong) * TR + it.lane;
    if (!one && (it.lane >= TR || nj >= d.n)) return;
    nv = !one || it.lane == 0;
    nb[0] = __ldg(d.H.rp + nj);
    ne[0] = __ldg(d.H.rp + nj + 1);
    nb[1] = __ldg(d.At.rp + nj);
    ne[1] = __ldg(d.At.rp + nj + 1);
    if (!LONG && !one && (ne[0] - nb[0] > kLongRowEntries || ne[1] - nb[1] > kLongRowEntries)) {
      nv = false;
      ne[0] = nb[0];
      ne[1] = nb[1];
    }
  };
  fetch(it.first);
  for (long long i = it.first; i < items; i += it.step) {
    const long long j = nj;
    const int rb[2] = {nb[0], nb[1]}, re[2] = {ne[0], ne[1]};
    const bool valid = nv;
    T xti = T(0), xci = T(0), hxc = T(0), atc = T(0), itx = T(0), xb = T(0), hb = T(0), qx = T(0), tau = T(0),
      lo = T(0), hi = T(0), sum[2];
    if (valid) {
      xti = xt[j];
      xci = xc[j];
      hxc = d.Hx[cur][j];
      atc = d.Aty[cur][j];
      itx = d.itaux[j];
      xb = d.xbar[a1][j];
      hb = d.Hxbar[a1][j];
      qx = d.qx[j];
      tau = d.taux[j];
      lo = d.lx[j];
      hi = d.ux[j];
    }
    fetch(i + it.step);
    if (LONG) {
      sum[0] = tile_long_rows<false, T>(ci[0], val[0], rb[0], re[0], f[0]);
      sum[1] = tile_long_rows<false, T>(ci[1], val[1], rb[1], re[1], f[1]);
    } else if (i < nlong) {
      sum[0] = warp_row<false, T>(ci[0], val[0], rb[0], re[0], f[0]);
      sum[1] = warp_row<false, T>(ci[1], val[1], rb[1], re[1], f[1]);
    } else {
      // FP32 gathers for both matrices together.  FP64, bound by its arithmetic,
      // takes them in turn: together 180 bytes of registers spill, and a call at
      // n = 200 takes 6.6 ms instead of 6.2, at n = 50,000 19.3 instead of 18.3, while
      // n = 1,000,000 gains 3 % (53.4 instead of 55.1).
      if (sizeof(T) == 4) {
        tile_rows<2, false, T, false>(ci, val, rb, re, f, buf, sum);
      } else {
        sum[0] = tile_rows1<false, T, false>(ci[0], val[0], rb[0], re[0], f[0], buf);
        sum[1] = tile_rows1<false, T, false>(ci[1], val[1], rb[1], re[1], f[1], buf);
      }
    }
    if (valid) {
      d.Hx[nx][j] = sum[0];
      d.Aty[nx][j] = sum[1];
      const T dx = xti - xci, dh = sum[0] - hxc, da = sum[1] - atc;
      ts.Lt += dx * dx * itx;
      ts.RH += fabs(dx) * fabs(dh);
      ts.RB += fabs(dx) * fabs(da);
      // The next trial's averages (weight alpha of this trial) and x_tr.
      hb = k0[kOma] * hb + k0[kAlpha] * sum[0];
      xb = k0[kOma] * xb + k0[kAlpha] * xti;
      d.Hxbar[a1 ^ 1][j] = hb;
      d.xbar[a1 ^ 1][j] = xb;
      const T g = qx + k0[kOma1] * hb + k0[kAlpha1] * sum[0] - sum[1];
      xs[j] = clampv<T>(xti - (k0[kSct] * tau) * g, lo, hi);
    }
  }
}

// This block's four sums to part[0..3] (fixed order): per warp the quantities
// are reduced together by halving (6 FP64 additions), then warp 0 adds the
// warps' sums.  Visible to the block after its next barrier.
__device__ __forceinline__ void block_sums(double (&v)[4], double *part) {
  __shared__ double ws[4][kTrialThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const bool hi = (lane & 16) != 0, lo = (lane & 8) != 0;
  double a0 = hi ? v[2] : v[0], a1 = hi ? v[3] : v[1];
  a0 += __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[2], 16);
  a1 += __shfl_xor_sync(0xffffffffu, hi ? v[1] : v[3], 16);
  double b = lo ? a1 : a0;
  b += __shfl_xor_sync(0xffffffffu, lo ? a0 : a1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
  if ((lane & 7) == 0) ws[lane >> 3][w] = b;  // quantity lane / 8
  __syncthreads();
  if (w == 0) {
    const int q = lane >> 3, i = lane & 7;
    b = i < nw ? ws[q][i] : 0.0;
    if (i + 8 < nw) b += ws[q][i + 8];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
    if (i == 0) part[q] = b;
  }
}

// Acceptance decision of the persistent loop, by the whole last block, on the
// block's own copy of the state: the blocks' sums (4 quantities, block-major)
// over 4 warps, then across lanes and warps in a fixed order.  Returns 1 when
// the loop goes on after an acceptance and nothing else: every block then
// makes the same change to its own copy (advance_trial); else 0, with the state
// in global memory for the others to load.  next: alpha of the trial after the
// next and beta after an acceptance.
__device__ __forceinline__ void advance_x(DevState *S) {
  const int x = S->xcur;
  S->xcur = S->xtr;
  S->xtr = S->xsp;
  S->xsp = x;
  S->spec = 1;
}
__device__ __forceinline__ void advance_trial(DevState *S, const double *next) {
  trial_begin(S);
  trial_accept(S);
  advance_x(S);
  advance_scalars(S, next[0], next[1]);
}
template <typename T>
__device__ __forceinline__ int decide_tiles(const Dev<T> &d, DevState &S, int nb, bool lr, const double *next,
                                            bool store = true) {
  __shared__ double red[4][4];
  __shared__ int go;
  const double *part = d.part + P_TRP * kMaxBlocks;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (w < 4) {
    double a = 0.0;
    if (nb == 1) {
      if (w == 0 && lane < 4) a = part[lane];
    } else {
#pragma unroll 5
      for (int b = w * 8 + (lane >> 2); b < nb; b += 32) a += __ldcg(part + 4 * b + (lane & 3));
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    }
    if (lane < 4) red[w][lane] = a;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      a[k] = (red[0][k] + red[1][k]) + (red[2][k] + red[3][k]);
      if (lr) a[k] += __ldcg(d.lr_acc + k);
    }
    const bool accepted = decide_logic(&S, a);
    if (accepted) {
      advance_x(&S);
      advance_scalars(&S, next[0], next[1]);
    } else {
      S.spec = 0;
      refresh_scalars(&S);
    }
    go = accepted && S.status == ST_RUNNING && S.slot_left > 0 && !S.check_due;
  }
  __syncthreads();
  if (!go && store) state_store(d.st, S);
  return go;
}

// Acceptance decision (single block, deterministic order).  On acceptance the
// trial buffers become current (index flip); on rejection both step vectors
// are shrunk through kappa.

// Acceptance decision (Eq. adaptive-condition), run by the last block of the
// column kernel once every block's partial sums are visible: FP64 sums in a
// fixed order; on acceptance the trial buffers become current (index flip), on
// rejection both step vectors shrink through kappa.  Sets the device-loop
// handles: hw (continue while running and the launch has trials left) and hc
// (a periodic check follows).
// The scalar part of the acceptance decision (one thread), from the sums of the
// trial over rows and columns: dw^2 / tau0, dy^2 / eta0, |dw'H dw| and |dw'B'dy|.
__device__ __forceinline__ bool accepts(const DevState *st, const double (&a)[4], bool &finite) {
  const double lhs = st->sd[kOka] * a[0] + st->sd[kIko] * a[1];
  finite = !nonfinite(lhs) && !nonfinite(a[2]) && !nonfinite(a[3]);
  return 0.5 * lhs >= 0.5 * a[2] + a[3];
}
// What every trial does to the state, and what an acceptance does (the x
// buffers are turned by the caller).
__device__ __forceinline__ void trial_begin(DevState *st) {
  // Commit the averages materialised by this trial's primal / row passes.
  st->acur ^= st->accepted;
  st->accepted = 0;
  st->restart_flag = 0;
  st->check_due = 0;
  st->trials += 1;
  st->slot_left -= 1;
}
__device__ __forceinline__ void trial_accept(DevState *st) {
  st->alpha_acc = st->sd[kAlpha];
  st->cur ^= 1;
  st->accepted = 1;
  st->t += 1;
  st->t_total += 1;
  st->accepted_all += 1;
  st->rej = 0;
}
__device__ __forceinline__ bool decide_logic(DevState *st, const double (&a)[4]) {
  bool finite;
  const bool ok = accepts(st, a, finite);
  trial_begin(st);
  if (!finite) {
    st->status = ST_NUMERICAL_ERROR;
    return false;
  }
  if (ok) {
    trial_accept(st);
    bool due = st->t_total == st->k_in;
    if (st->k_chk > 0)
      due |= ((st->t_total | st->k_chk) >> 32) == 0 ? (unsigned)st->t_total % (unsigned)st->k_chk == 0
                                                     : st->t_total % st->k_chk == 0;
    st->check_due = due ? 1 : 0;
    if (!due && st->t_total == st->pause_at) st->status = ST_PAUSED;
    return true;
  }
  st->kappa *= st->shrink;
  st->rej += 1;
  if (st->rej >= st->rej_limit) st->status = ST_NUMERICAL_ERROR;
  return false;
}

template <bool COND>
__device__ void decide_body(DevState *stg, const double *part, const double *lacc, int nb_r, int nb_c,
                            cudaGraphConditionalHandle hw, cudaGraphConditionalHandle hc) {
  __shared__ DevState S;
  state_load(S, stg);
  double a[4], b[4];
  if (nb_r == nb_c) {
    // Row and column partials of one grid (rows 0-3 and 4-7): one pass.
    double ab[8];
    final_reduce<8>(part + P_TR_R * kMaxBlocks, nb_r, 0u, ab);
    for (int k = 0; k < 4; ++k) {
      a[k] = ab[k];
      b[k] = ab[4 + k];
    }
  } else {
    final_reduce<4>(part + P_TR_R * kMaxBlocks, nb_r, 0u, a);
    final_reduce<4>(part + P_TR_C * kMaxBlocks, nb_c, 0u, b);
  }
  if (lacc)
    for (int k = 0; k < 4; ++k) a[k] += __ldcg(lacc + k);
  if (threadIdx.x == 0) {
    for (int k = 0; k < 4; ++k) a[k] += b[k];
    if (decide_logic(&S, a)) {
      const int x = S.xcur;
      S.xcur = S.xtr;
      S.xtr = x;
    }
    refresh_scalars(&S);
    if (COND) {
      const bool run = S.status == ST_RUNNING;
      if (hw) cudaGraphSetConditional(hw, (run && S.slot_left > 0) ? 1u : 0u);
      if (hc) cudaGraphSetConditional(hc, (run && S.check_due) ? 1u : 0u);
    }
  }
  state_store(stg, S);
}

// Materialises the running averages of a pending acceptance: bar[acur^1] =
// (1 - alpha) bar[acur] + alpha w (Algorithm 4, "update the weighted
// averages") for x, H x, s, r, y.  The trial kernels do this lazily; this
// kernel is only used before the host reads a paused state.  Reads and writes
// different buffers, so a repeated launch is harmless.
template <typename T>
__global__ void __launch_bounds__(kBlock) k_average(Dev<T> d) {
  const DevState *st = d.st;
  if (!st->accepted) return;
  const int cur = st->cur, a0 = st->acur, a1 = st->acur ^ 1;
  const T alpha = T(st->alpha_acc), oma = T(1) - alpha;
  PDNQP_GRID_STRIDE(i, d.n) {
    d.xbar[a1][i] = oma * d.xbar[a0][i] + alpha * d.x[st->xcur][i];
    d.Hxbar[a1][i] = oma * d.Hxbar[a0][i] + alpha * d.Hx[cur][i];
  }
  PDNQP_GRID_STRIDE(j, d.m) {
    d.ybar[a1][j] = oma * d.ybar[a0][j] + alpha * d.y[cur][j];
    d.rbar[a1][j] = oma * d.rbar[a0][j] + alpha * d.r[cur][j];
    if (j >= d.mE) d.sbar[a1][j] = oma * d.sbar[a0][j] + alpha * d.s[cur][j];
  }
}

// ===========================================================================
// Periodic check (Sec. 3.3.3 inner termination; restart criteria and the
// primal weight, Eqs. primal-weight-movement / primal-weight-update).
// Per candidate (c = current, a = average) 8 quantities:
//   0 r_p (max), 1 s_p (max), 2 r_d (max), 3 s_d (max),
//   4 sum (d (Bw - h))^2, 5 sum ((w - P(w - e^2 g)) / e)^2,
//   6 sum ((w - w_start) / e)^2, 7 sum ((y - y_start) / d)^2
// stored as [c0..c7, a0..a7].
// ===========================================================================
// Contributions of one row (its s and r components and its dual) to the 8
// quantities of one candidate, in FP64.  Inputs are corrections (bwd = B dw,
// ds, dr, dy, epoch-start corrections) plus the base data of the row.
struct RowIn {
  bool ineq;
  double bwd, hp, bwb, h;        // B dw, h - B w_b, B w_b, h
  double ds, dr, dyv;            // corrections
  double qs, qr, sig, lam;       // base gradients (s, r blocks), penalty, multiplier
  double rb, yb;                 // base r and y
  double ls, us;                 // shifted slack bounds
  double es, er, dsc;            // column scales of s, r and the row scale
  double ies, ier, idsc;         // their reciprocals
  double sst, rst, yst;          // epoch-start corrections
};

__device__ __forceinline__ void row_cand(double *q, const RowIn &a) {
  const double e_bh = a.bwd - a.hp;  // (B w - h)_j
  q[0] = max_abs(q[0], e_bh);
  q[1] = max_abs(max_abs(q[1], a.bwb + a.bwd), a.h);
  const double gr = a.qr + a.sig * a.dr + a.dyv;  // sigma r + lambda + y at the point
  q[2] = max_abs(q[2], gr);
  q[3] = max_abs(max_abs(max_abs(q[3], a.sig * (a.rb + a.dr)), a.lam), a.yb + a.dyv);
  const double eb = a.dsc * e_bh, eg = a.er * gr;
  q[4] += eb * eb;
  q[5] += eg * eg;
  const double wr = (a.dr - a.rst) * a.ier;
  q[6] += wr * wr;
  const double wy = (a.dyv - a.yst) * a.idsc;
  q[7] += wy * wy;
  if (a.ineq) {
    const double gs = a.qs + a.dyv;  // y at the point
    q[2] = max_abs(q[2], a.ds - clampv<double>(a.ds - gs, a.ls, a.us));
    const double ks = (a.ds - clampv<double>(a.ds - a.es * a.es * gs, a.ls, a.us)) * a.ies;
    q[5] += ks * ks;
    const double ws = (a.ds - a.sst) * a.ies;
    q[6] += ws * ws;
  }
}

template <typename T, int G>
__device__ __forceinline__ void check_rows_body(const Dev<T> &d, const DevState *st, GridCtx g,
                                                Slot<T> *buf) {
  // Averages of a pending acceptance are formed on the fly (and written for the
  // row blocks); x bar is gathered as (1 - alpha) xbar + alpha x.
  const int cur = st->cur, a0 = st->acur, acc = st->accepted, ab = a0 ^ acc;
  const T ap = T(st->alpha_acc), omap = T(1) - ap;
  const T *xb0 = d.xbar[a0];
  const T *xc = d.x[st->xcur];
  double q[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) q[k] = 0.0;
  TileIter<G> ti(g);
  for (long long tile = ti.first; tile < d.m; tile += ti.step) {
    const T axb = tile_row_sum<G, T>(d.A.rp, d.A.ci, d.A.val, tile, d.m,
                               entry([&](int k) { return acc ? omap * xb0[k] + ap * xc[k] : xb0[k]; }, AddProduct()), buf);
    long long j;
    const bool own = ti.row(tile, d.m, j);
    if (own) {
      const bool ineq = j >= d.mE;
      RowIn a;
      a.ineq = ineq;
      a.hp = widen(d.hp[j]);
      a.bwb = widen(d.Bwb[j]);
      a.h = widen(d.h[j]);
      a.qs = ineq ? widen(d.qs[j]) : 0.0;
      a.qr = widen(d.qr[j]);
      a.sig = d.sig[j];
      a.lam = d.lam[j];
      a.rb = d.rb[j];
      a.yb = d.yb[j];
      a.ls = ineq ? widen(d.ls[j]) : 0.0;
      a.us = ineq ? widen(d.us[j]) : 0.0;
      a.es = ineq ? widen(d.es[j]) : 1.0;
      a.er = widen(d.er[j]);
      a.dsc = widen(d.dy[j]);
      a.ies = ineq ? recip(d.es[j]) : 1.0;
      a.ier = recip(d.er[j]);
      a.idsc = recip(d.dy[j]);
      a.sst = ineq ? widen(d.sst[j]) : 0.0;
      a.rst = widen(d.rst[j]);
      a.yst = widen(d.yst[j]);
      a.bwd = widen(d.Bw[cur][j]);
      a.ds = ineq ? widen(d.s[cur][j]) : 0.0;
      a.dr = widen(d.r[cur][j]);
      a.dyv = widen(d.y[cur][j]);
      row_cand(q, a);
      {
        T sa = ineq ? d.sbar[a0][j] : T(0), ra = d.rbar[a0][j], ya = d.ybar[a0][j];
        if (acc) {
          ra = omap * ra + ap * d.r[cur][j];
          ya = omap * ya + ap * d.y[cur][j];
          d.rbar[ab][j] = ra;
          d.ybar[ab][j] = ya;
          if (ineq) {
            sa = omap * sa + ap * d.s[cur][j];
            d.sbar[ab][j] = sa;
          }
        }
        const T bwa = axb - sa - ra;
        d.Bwbar[j] = bwa;
        a.bwd = widen(bwa);
        a.ds = widen(sa);
        a.dr = widen(ra);
        a.dyv = widen(ya);
        row_cand(q + 8, a);
      }
    }
  }
  block_reduce_store<16, CK_MAXMASK>(q, d.part + P_CK_R * kMaxBlocks, g.b);
}

template <typename T>
__device__ __forceinline__ bool check_pending(const Dev<T> &d) {
  return d.st->status == ST_RUNNING && d.st->check_due;
}

template <typename T, int G>
__global__ void __launch_bounds__(kBlock) k_check_rows(Dev<T> d) {
  if (!check_pending(d)) return;
  check_rows_body<T, G>(d, d.st, hw_grid(), warp_slots<T>());
}

// Contributions of one variable (x block) to the 8 quantities of a candidate:
// dx, H dx, A' dy corrections plus the base data of the variable.
__device__ __forceinline__ void col_cand(double *q, double dx, double hdx, double atdy, double qx, double qx0,
                                         double hxb, double atyb, double lx, double ux, double ex2, double iex,
                                         double xst) {
  const double g = hdx + qx - atdy;  // gradient of the inner Lagrangian at the point
  q[2] = max_abs(q[2], dx - clampv<double>(dx - g, lx, ux));
  q[3] = max_abs(max_abs(max_abs(q[3], hxb + hdx), qx0), atyb + atdy);
  const double k = (dx - clampv<double>(dx - ex2 * g, lx, ux)) * iex;
  q[5] += k * k;
  const double w = (dx - xst) * iex;
  q[6] += w * w;
}

template <typename T, int G>
__device__ __forceinline__ void check_cols_terms(const Dev<T> &d, const DevState *st, GridCtx g,
                                                 Slot<T> *buf) {
  // y bar of a pending acceptance was materialised by k_check_rows.
  const int cur = st->cur, a0 = st->acur, acc = st->accepted, ab = a0 ^ acc;
  const T ap = T(st->alpha_acc), omap = T(1) - ap;
  const T *yb = d.ybar[ab];
  const T *xc = d.x[st->xcur];
  double q[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) q[k] = 0.0;
  TileIter<G> ti(g);
  for (long long tile = ti.first; tile < d.n; tile += ti.step) {
    const T atyb = tile_row_sum<G, T>(d.At.rp, d.At.ci, d.At.val, tile, d.n, MulLd<T>{yb}, buf);
    long long i;
    const bool own = ti.row(tile, d.n, i);
    if (own) {
      const double qx = widen(d.qx[i]), qx0 = widen(d.qx0[i]), hxb = widen(d.Hxb[i]);
      const double atyb0 = widen(d.Atyb[i]), lx = widen(d.lx[i]), ux = widen(d.ux[i]);
      const double ex = widen(d.ex[i]), xst = widen(d.xst[i]), iex = recip(d.ex[i]), ex2 = ex * ex;
      col_cand(q, widen(xc[i]), widen(d.Hx[cur][i]), widen(d.Aty[cur][i]), qx, qx0, hxb, atyb0, lx, ux, ex2, iex, xst);
      {
        d.Atybar[i] = atyb;
        T xa = d.xbar[a0][i], ha = d.Hxbar[a0][i];
        if (acc) {
          xa = omap * xa + ap * xc[i];
          ha = omap * ha + ap * d.Hx[cur][i];
          d.xbar[ab][i] = xa;
          d.Hxbar[ab][i] = ha;
        }
        col_cand(q + 8, widen(xa), widen(ha), widen(atyb), qx, qx0, hxb, atyb0, lx, ux, ex2, iex, xst);
      }
    }
  }
  block_reduce_store<16, CK_MAXMASK>(q, d.part + P_CK_C * kMaxBlocks, g.b);
}

template <typename T, int G, bool COND>
__device__ __forceinline__ void check_cols_body(const Dev<T> &d, int nb_r, GridCtx g) {
  if (!check_pending(d)) return;
  check_cols_terms<T, G>(d, d.st, g, warp_slots<T>());
  if (arrive_last(d.ctr + 1, g.nb)) {
    check_final_body<COND>(d.st, d.part, nb_r, g.nb, d.hw);
    if (threadIdx.x == 0) d.ctr[1] = 0u;
  }
}

template <typename T, int G, bool COND>
__global__ void __launch_bounds__(kBlock) k_check_cols(Dev<T> d, int nb_r) {
  check_cols_body<T, G, COND>(d, nb_r, hw_grid());
}

// Decisions of the check (one thread), from its 16 quantities: inner termination
// of both candidates (Eq. inner-termination), iteration limit, restart criteria
// and primal weight.
__device__ __forceinline__ void check_logic(DevState *st, const double (&q)[16]) {
  for (int k = 0; k < 16; ++k) st->chk[k] = q[k];
  // The averages of this trial's acceptance were materialised by the check's
  // passes.  The check is consumed here; the restart itself is applied by
  // check_apply_body on restart_flag.
  st->acur ^= st->accepted;
  st->accepted = 0;
  st->restart_flag = 0;
  st->check_due = 0;
  const double dta = st->dta, dtr = st->dtr;
  const double spc = fmax(1.0, q[1]), sdc = fmax(1.0, q[3]);
  const double spa = fmax(1.0, q[9]), sda = fmax(1.0, q[11]);
  const bool okc = q[0] <= dta + dtr * spc && q[2] <= dta + dtr * sdc;
  const bool oka = q[8] <= dta + dtr * spa && q[10] <= dta + dtr * sda;
  if (!st->ignore_conv && okc) {
    st->status = ST_CONVERGED;
    st->ret_avg = 0;
  } else if (!st->ignore_conv && oka) {
    st->status = ST_CONVERGED;
    st->ret_avg = 1;
  } else if (st->t_total == st->k_in) {
    st->status = ST_ITER_LIMIT;
  } else {
    const double om = st->omega;
    const double kc = sqrt(om * q[4] + q[5] / om);
    const double ka = sqrt(om * q[12] + q[13] / om);
    const bool use_avg = ka < kc;
    const double kcand = use_avg ? ka : kc;
    const bool restart = kcand <= st->beta_suff * st->k_restart ||
                         (kcand <= st->beta_nec * st->k_restart && kcand > st->k_last) ||
                         (double)st->t >= st->beta_art * (double)st->t_total;
    st->k_last = kcand;
    if (restart) {
      const double dW = sqrt(use_avg ? q[14] : q[6]);
      const double dY = sqrt(use_avg ? q[15] : q[7]);
      if (dW > 0.0 && dY > 0.0) st->omega = exp(0.25 * log(dY / dW) + 0.75 * log(om));
      st->kappa = 1.0;
      st->t = 0;
      st->k_restart = kcand;
      st->k_last = INFINITY;
      st->restarts += 1;
      st->restart_flag = 1;
      st->spec = 0;
      st->restart_use_avg = use_avg ? 1 : 0;
    }
    if (st->t_total == st->pause_at) st->status = ST_PAUSED;
  }
  refresh_scalars(st);
}
// The quantities of a check from the row and column partials (whole block).
__device__ __forceinline__ void check_sums(const double *part, int nb_r, int nb_c, double (&q)[16]) {
  double b[16];
  final_reduce<16>(part + P_CK_R * kMaxBlocks, nb_r, CK_MAXMASK, q);
  final_reduce<16>(part + P_CK_C * kMaxBlocks, nb_c, CK_MAXMASK, b);
#pragma unroll
  for (int k = 0; k < 16; ++k) q[k] = ((CK_MAXMASK >> k) & 1u) ? fmax(q[k], b[k]) : q[k] + b[k];
}

template <bool COND>
__device__ void check_final_body(DevState *stg, const double *part, int nb_r, int nb_c,
                                 cudaGraphConditionalHandle hw) {
  __shared__ DevState S;
  state_load(S, stg);
  double q[16];
  check_sums(part, nb_r, nb_c, q);
  if (threadIdx.x == 0) {
    check_logic(&S, q);
    if (COND && hw) cudaGraphSetConditional(hw, (S.status == ST_RUNNING && S.slot_left > 0) ? 1u : 0u);
  }
  state_store(stg, S);
}

// Restart (Algorithm 4): optionally move the current point to the average
// (with its cached products), then make it the epoch start and clear the
// averages.  Idempotent, so a repeated launch is harmless.
template <typename T>
__device__ __forceinline__ void check_apply_body(const Dev<T> &d, const DevState *st, GridCtx g) {
  if (!st->restart_flag) return;
  const int cur = st->cur, ab = st->acur;
  const bool ua = st->restart_use_avg;
  T *xc = d.x[st->xcur];
  PDNQP_VGRID_STRIDE(i, d.n, g) {
    T x = xc[i], hx = d.Hx[cur][i];
    if (ua) {
      x = d.xbar[ab][i];
      hx = d.Hxbar[ab][i];
      xc[i] = x;
      d.Hx[cur][i] = hx;
      d.Aty[cur][i] = d.Atybar[i];
    }
    d.xst[i] = x;
    d.xbar[ab][i] = x;
    d.Hxbar[ab][i] = hx;
  }
  PDNQP_VGRID_STRIDE(j, d.m, g) {
    T y = d.y[cur][j], r = d.r[cur][j];
    if (ua) {
      y = d.ybar[ab][j];
      r = d.rbar[ab][j];
      d.y[cur][j] = y;
      d.r[cur][j] = r;
      d.Bw[cur][j] = d.Bwbar[j];
    }
    d.yst[j] = y;
    d.rst[j] = r;
    d.ybar[ab][j] = y;
    d.rbar[ab][j] = r;
    if (j >= d.mE) {
      T s = d.s[cur][j];
      if (ua) {
        s = d.sbar[ab][j];
        d.s[cur][j] = s;
      }
      d.sst[j] = s;
      d.sbar[ab][j] = s;
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(kBlock) k_check_apply(Dev<T> d) {
  check_apply_body<T>(d, d.st, hw_grid());
}

// ===========================================================================
// The persistent loop.
// ===========================================================================
// Persistent trial loop (one cooperative launch).  A trial is the row pass, a
// grid barrier, the column pass (with the next trial's primal step) and a grid
// barrier whose last block takes the acceptance decision; a trial whose primal
// step is not there yet (the first one, after a rejection, after a restart)
// starts with the primal pass and a barrier.  The loop leaves when the solve
// stops, a periodic check is due (k_check follows this launch; in this kernel
// its FP64 terms would take registers from the passes, 62.7 instead of 54 us for
// the FP64 row pass at n = 1e6) or the trial allowance is used up (chunk >= 0
// sets it); it does not start while a check is pending.  All blocks take the same
// branches (the state is block-uniform), so every barrier is reached by every
// block.  LR: the instance has dense coupling rows (d.nlr > 0); RL / CL:
// long rows of A / of H and A' (tiles of 8).
template <typename T, bool LR, bool RL, bool CL, bool CLU>
__global__ void __launch_bounds__(kTrialThreads, 1) k_trials(Dev<T> d, long long chunk) {
  __shared__ DevState S;
  __shared__ double next[2];
  extern __shared__ __align__(16) unsigned char slots[];
  Slot<T> *buf = reinterpret_cast<Slot<T> *>(slots) + (threadIdx.x >> 5) * kTileSlots;
  unsigned *bar = d.ctr + kCtrBar;
  unsigned gen = threadIdx.x == 0 ? ld_acquire_gpu(bar + kBarGen) : 0u;
  state_load(S, d.st);
  if (threadIdx.x == 0 && chunk >= 0) S.slot_left = chunk;
  __syncthreads();
  const int nb = gridDim.x;
  double *part = d.part + P_TRP * kMaxBlocks + 4 * blockIdx.x;
  // Block 0 times each pass: its own work, then its wait at the barrier
  // (imbalance across blocks plus the barrier itself; the last one includes
  // the acceptance decision).
  const bool timer = blockIdx.x == 0 && threadIdx.x == 0;
  unsigned long long tp[6] = {0ull, 0ull, 0ull, 0ull, 0ull, 0ull};
  unsigned long long tk = timer ? global_ns() : 0ull;
  auto lap = [&](int k) {
    if (timer) {
      const unsigned long long t = global_ns();
      tp[k] += t - tk;
      tk = t;
    }
  };
  while (S.status == ST_RUNNING && S.slot_left > 0 && !S.check_due) {
    if (!S.spec) {
      primal_phase<T>(d, &S);
      lap(0);
      if (loop_sync<CLU, false>(bar, gen) < 0) return;
      lap(1);
    }
    if (threadIdx.x >= kTrialThreads - 2) {  // a spare lane each, before the last warp's first item
      const double t = (double)(S.t + 1);
      if (threadIdx.x == kTrialThreads - 2)
        next[0] = 2.0 / (t + 3.0);
      else
        next[1] = t / (t + 1.0);
    }
    TrialSums<T> ts = {T(0), T(0), T(0), T(0)};
    rows_phase_tiles<T, LR, RL>(d, &S, buf, ts);
    lap(2);
    if (LR) {
      if (loop_sync<CLU, false>(bar, gen, [&] {
            long_rows_finish<T>(d, &S, d.lr_nb);
            return 0;
          }) < 0)
        return;
    } else if (loop_sync<CLU, false>(bar, gen) < 0) {
      return;
    }
    lap(3);
    cols_phase_tiles<T, CL>(d, &S, buf, ts);
    lap(4);
    double v[4] = {widen(ts.Lt), widen(ts.Le), widen(ts.RH), widen(ts.RB)};
    block_sums(v, part);
    bool led = CLU;
    int go;
    if (CLU) {  // every block of a cluster decides for itself, on the same sums
      loop_sync<CLU, false>(bar, gen);
      go = decide_tiles<T>(d, S, nb, LR, next, blockIdx.x == 0);
    } else {
      go = loop_sync<CLU, false>(bar, gen, [&] {
        led = true;
        return decide_tiles<T>(d, S, nb, LR, next);
      });
    }
    if (go < 0) return;
    if (!led) {
      if (go) {
        if (threadIdx.x == 0) advance_trial(&S, next);
        __syncthreads();
      } else {
        state_load(S, d.st);
      }
    }
    lap(5);
  }
  if (timer && d.ptime)
    for (int k = 0; k < 6; ++k) d.ptime[k] += tp[k];
}

// Periodic check of the persistent form, with its restart, in one cooperative
// launch on the loop's grid: the two passes, the decision in the last block of
// the second barrier, and the restart.  Does nothing when no check is pending.
template <typename T, bool RL, bool CL, bool CLU>
__global__ void __launch_bounds__(kTrialThreads, 1) k_check(Dev<T> d) {
  __shared__ DevState S;
  extern __shared__ __align__(16) unsigned char slots[];
  Slot<T> *buf = reinterpret_cast<Slot<T> *>(slots) + (threadIdx.x >> 5) * kTileSlots;
  unsigned *bar = d.ctr + kCtrBar;
  unsigned gen = threadIdx.x == 0 ? ld_acquire_gpu(bar + kBarGen) : 0u;
  state_load(S, d.st);
  if (S.status != ST_RUNNING || !S.check_due) return;
  const int nb = gridDim.x;
  const GridCtx g{(int)blockIdx.x, nb};
  check_rows_body<T, RL ? 16 : 8>(d, &S, g, buf);
  if (loop_sync<CLU>(bar, gen) < 0) return;
  check_cols_terms<T, CL ? 16 : 8>(d, &S, g, buf);
  bool led = false;
  if (loop_sync<CLU>(bar, gen, [&] {
        led = true;
        double q[16];
        check_sums(d.part, nb, nb, q);
        if (threadIdx.x == 0) check_logic(&S, q);
        state_store(d.st, S);
        return 0;
      }) < 0)
    return;
  if (!led) state_load(S, d.st);
  check_apply_body<T>(d, &S, g);
}

// End of an inner solve: the outer x and inner y become base + correction
// (the current point, or the average when it is the converged candidate), and
// dx = x - x_prev over the outer iteration (infeasibility tests).
template <typename T>
__global__ void k_finish(Dev<T> d, double *x64, double *y64, const double *xprev, double *dxv, int use_avg) {
  const int cur = d.st->cur, ab = d.st->acur ^ d.st->accepted;
  const T *__restrict__ dx = use_avg ? d.xbar[ab] : d.x[d.st->xcur];
  const T *__restrict__ dy = use_avg ? d.ybar[ab] : d.y[cur];
  PDNQP_GRID_STRIDE(i, d.n) {
    const double x = x64[i] + double(dx[i]);
    x64[i] = x;
    dxv[i] = x - xprev[i];
  }
  PDNQP_GRID_STRIDE(j, d.m) y64[j] += double(dy[j]);
}

// Totals of the current and averaged points for a snapshot:
// out = [w (dw) | y (m) | wbar (dw) | ybar (m)], w = (x, s_I, r_E, r_I).
template <typename T>
__global__ void k_totals(Dev<T> d, double *out) {
  const int cur = d.st->cur, ab = d.st->acur ^ d.st->accepted;
  const long long n = d.n, m = d.m, mI = m - d.mE, dw = n + mI + m;
  for (int a = 0; a < 2; ++a) {
    const T *x = a ? d.xbar[ab] : d.x[d.st->xcur];
    const T *s = a ? d.sbar[ab] : d.s[cur];
    const T *r = a ? d.rbar[ab] : d.r[cur];
    const T *y = a ? d.ybar[ab] : d.y[cur];
    double *o = out + a * (dw + m);
    PDNQP_GRID_STRIDE(i, n) o[i] = d.xb[i] + double(x[i]);
    PDNQP_GRID_STRIDE(j, m) {
      if (j >= d.mE) o[n + (j - d.mE)] = d.sb[j] + double(s[j]);
      o[n + mI + j] = d.rb[j] + double(r[j]);
      o[dw + j] = d.yb[j] + double(y[j]);
    }
  }
}

// ===========================================================================
// Batched form: the inner iterations of many problems in one launch per
// phase.  Block k of a batched launch works for problem map[k].p as block
// map[k].b of map[k].nb (the problem's own partition, the same as when it
// runs alone, so its reductions and its iterates are bitwise those of its
// solo graph-form solve); the problem's device pointers come from devs[p].
// Every phase skips a problem whose status is not ST_RUNNING, so problems
// that wait for their host outer iteration cost one state read per block; the
// trial phases also skip one whose periodic check is due.
// ===========================================================================
struct BatchBlk {
  int p, b, nb;
};

// The problem's Dev copied to shared memory once per block (its pointers are
// then read without a global-memory round trip per use).
template <typename T>
__device__ __forceinline__ const Dev<T> &batch_dev(const Dev<T> *devs, int p) {
  __shared__ __align__(16) unsigned char buf[sizeof(Dev<T>)];
  static_assert(sizeof(Dev<T>) % 4 == 0, "Dev must be a whole number of words");
  const int *src = reinterpret_cast<const int *>(devs + p);
  for (int i = threadIdx.x; i < (int)(sizeof(Dev<T>) / 4); i += blockDim.x) reinterpret_cast<int *>(buf)[i] = src[i];
  __syncthreads();
  return *reinterpret_cast<const Dev<T> *>(buf);
}

template <typename T>
__global__ void __launch_bounds__(kBlock) kb_primal(const Dev<T> *devs, const BatchBlk *map) {
  const BatchBlk e = map[blockIdx.x];
  const Dev<T> &d = batch_dev(devs, e.p);
  if (d.st->status != ST_RUNNING || d.st->check_due) return;
  primal_phase<T>(d, d.st, GridCtx{e.b, e.nb});
}

template <typename T, int G>
__global__ void __launch_bounds__(kBlock) kb_rows(const Dev<T> *devs, const BatchBlk *map) {
  const BatchBlk e = map[blockIdx.x];
  rows_trial_body<T, G>(batch_dev(devs, e.p), GridCtx{e.b, e.nb});
}

// nb_rows[p]: blocks of problem p in the row launches (its row partials).
template <typename T, int G>
__global__ void __launch_bounds__(kBlock) kb_cols(const Dev<T> *devs, const BatchBlk *map, const int *nb_rows) {
  const BatchBlk e = map[blockIdx.x];
  cols_trial_body<T, G, false>(batch_dev(devs, e.p), nb_rows[e.p], GridCtx{e.b, e.nb});
}

template <typename T, int G>
__global__ void __launch_bounds__(kBlock) kb_check_rows(const Dev<T> *devs, const BatchBlk *map) {
  const BatchBlk e = map[blockIdx.x];
  const Dev<T> &d = batch_dev(devs, e.p);
  if (!check_pending(d)) return;
  check_rows_body<T, G>(d, d.st, GridCtx{e.b, e.nb}, warp_slots<T>());
}

template <typename T, int G>
__global__ void __launch_bounds__(kBlock) kb_check_cols(const Dev<T> *devs, const BatchBlk *map,
                                                        const int *nb_rows) {
  const BatchBlk e = map[blockIdx.x];
  check_cols_body<T, G, false>(batch_dev(devs, e.p), nb_rows[e.p], GridCtx{e.b, e.nb});
}

template <typename T>
__global__ void __launch_bounds__(kBlock) kb_check_apply(const Dev<T> *devs, const BatchBlk *map) {
  const BatchBlk e = map[blockIdx.x];
  const Dev<T> &d = batch_dev(devs, e.p);
  check_apply_body<T>(d, d.st, GridCtx{e.b, e.nb});
}

// Every problem idle, before the first graph launch: the graph runs as soon as one
// problem is set up, when the host threads of others have not reached theirs yet,
// and a handle may come from a debug run, which leaves its state running.
template <typename T>
__global__ void kb_idle(const Dev<T> *devs, int count) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < count; k += gridDim.x * blockDim.x)
    devs[k].st->status = ST_IDLE;
}

// Scheduler edits between graph launches: problems in `go` that are set up
// (ST_READY) start running; problems in `stop` that still run pause (their
// time limit passed).
template <typename T>
__global__ void kb_control(const Dev<T> *devs, const int *go, int ngo, const int *stop, int nstop) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < ngo + nstop; k += gridDim.x * blockDim.x) {
    DevState *st = devs[k < ngo ? go[k] : stop[k - ngo]].st;
    if (k < ngo) {
      if (st->status == ST_READY) st->status = ST_RUNNING;
    } else if (st->status == ST_RUNNING) {
      st->status = ST_PAUSED;
    }
  }
}

// Copies every problem's device state into one array (one read-back per launch).
template <typename T>
__global__ void kb_gather_states(const Dev<T> *devs, int count, DevState *out) {
  constexpr int W = (int)(sizeof(DevState) / 4);
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < (long long)count * W;
       k += (long long)gridDim.x * blockDim.x) {
    const int p = (int)(k / W), w = (int)(k % W);
    reinterpret_cast<int *>(out + p)[w] = __ldcg(reinterpret_cast<const int *>(devs[p].st) + w);
  }
}

}  // namespace
}  // namespace pdq

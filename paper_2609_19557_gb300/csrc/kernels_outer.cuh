// Kernels of the one-time setup (Sec. 3.1: outer Ruiz scaling, objective
// scalar, Lanczos estimate for gamma, initial penalties) and of the outer
// glue of Algorithm 3 (Eqs. practical-multiplier-update, outer-residuals,
// outer-scales, penalty-trigger-eq).  All of them compute in FP64.
#pragma once
#include <math.h>
#include <stdint.h>

#include "common.cuh"
#include "kernels.cuh"

namespace pdq {
namespace {  // internal linkage: each solver TU owns its kernels

// ---------------------------------------------------------------------------
// Outer Ruiz scaling of [[Q, A^T], [A, 0]] (Eq. scaled-problem).
// ---------------------------------------------------------------------------
template <int G>
__global__ void __launch_bounds__(kBlock) k_oruiz_rows(Mat<double> A, const double *Dc, const double *Dx, double *rn) {
  TileIter<G> ti;
  for (long long tile = ti.first; tile < A.nrows; tile += ti.step) {
    long long j;
    const bool own = ti.row(tile, A.nrows, j);
    const double a = tile_row_max<G, double>(A.rp, A.ci, A.val, tile, A.nrows, entry([&](int k) { return Dx[k]; }, MaxAbs()));
    if (own) rn[j] = a * Dc[j];
  }
}

template <int G>
__global__ void __launch_bounds__(kBlock) k_oruiz_cols(Mat<double> At, Mat<double> Q, const double *Dc,
                                                       const double *Dx, double *cn) {
  TileIter<G> ti;
  for (long long tile = ti.first; tile < Q.nrows; tile += ti.step) {
    long long i;
    const bool own = ti.row(tile, Q.nrows, i);
    const double a = tile_row_max<G, double>(At.rp, At.ci, At.val, tile, Q.nrows, entry([&](int k) { return Dc[k]; }, MaxAbs()));
    const double b = tile_row_max<G, double>(Q.rp, Q.ci, Q.val, tile, Q.nrows, entry([&](int k) { return Dx[k]; }, MaxAbs()));
    if (own) cn[i] = max_abs(a, b) * Dx[i];
  }
}

__global__ void k_ruiz_apply(double *D, const double *nrm, long long len) {
  PDNQP_GRID_STRIDE(i, len) {
    const double c = nrm[i];
    if (c > 0.0) D[i] = D[i] * (1.0 / sqrt(c));
  }
}

// val_k *= mult * rs[row] * cs[col] (a warp per row)
__global__ void k_scale_csr(int nrows, const int *rp, const int *ci, double *val, const double *rs, const double *cs,
                            double mult) {
  const int lane = threadIdx.x & 31;
  for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < nrows;
       i += ((long long)gridDim.x * blockDim.x) >> 5) {
    const double ri = rs[i] * mult;
    for (unsigned k = rp[i] + lane, e = rp[i + 1]; k < e; k += 32) val[k] = ri * val[k] * cs[ci[k]];
  }
}

// Max absolute row sum (induced l_inf norm) partials of a CSR matrix.
template <int G>
__global__ void __launch_bounds__(kBlock) k_rowabs_max(Mat<double> M, double *part) {
  double best = 0.0;
  TileIter<G> ti;
  for (long long tile = ti.first; tile < M.nrows; tile += ti.step)
    best = max_abs(best, tile_row_sum<G, double>(M.rp, M.ci, M.val, tile, M.nrows, entry([](int) { return 1.0; }, AddAbs())));
  double v[1] = {best};
  block_reduce_store<1, 1u>(v, part);
}

__global__ void k_absmax(const double *v, long long n, double *part) {
  double best = 0.0;
  PDNQP_GRID_STRIDE(i, n) best = fmax(best, fabs(v[i]));
  double q[1] = {best};
  block_reduce_store<1, 1u>(q, part);
}

// Reduction of nq quantities (row q of part, nb partials each) -> out[q]:
// block q reduces quantity q (fixed order: lane-strided serial sums, then a
// serial sum of the 32 lane sums).
__global__ void __launch_bounds__(32) k_reduce_rows(const double *part, int nq, int nb, unsigned max_mask, double *out) {
  __shared__ double ls[32];
  const int q = blockIdx.x, lane = threadIdx.x;
  if (q >= nq) return;
  const bool mx = q < 32 && ((max_mask >> q) & 1u);
  double a = 0.0;
  for (int b = lane; b < nb; b += 32) {
    const double p = part[(long long)q * kMaxBlocks + b];
    a = mx ? fmax(a, p) : a + p;
  }
  ls[lane] = a;
  __syncwarp();
  if (lane == 0) {
    double r = ls[0];
    for (int k = 1; k < 32; ++k) r = mx ? fmax(r, ls[k]) : r + ls[k];
    out[q] = r;
  }
}

// Diagonal shift: val[diag[i]] += s (diag[i] = position of (i, i) in row i).
__global__ void k_add_diag(int n, const int *diag, double *val, double s) {
  PDNQP_GRID_STRIDE(i, n) val[diag[i]] += s;
}

__global__ void k_scale_vec(double *v, const double *by, long long n, int divide, double mult) {
  PDNQP_GRID_STRIDE(i, n) v[i] = (divide ? v[i] / by[i] : v[i] * by[i]) * mult;
}

template <typename T>
__global__ void k_to_T(T *dst, const double *src, long long n) {
  PDNQP_GRID_STRIDE(i, n) dst[i] = T(src[i]);
}
__global__ void k_fill_d(double *p, long long n, double v) {
  PDNQP_GRID_STRIDE(i, n) p[i] = v;
}
__global__ void k_mul_scalar(double *p, long long n, double a) {
  PDNQP_GRID_STRIDE(i, n) p[i] *= a;
}
// ---------------------------------------------------------------------------
// Lanczos (Eq. R-choice): both starts together, in one cooperative launch or in a
// launch per phase.
// ---------------------------------------------------------------------------
// i-th output of the splitmix64 generator seeded with `seed`, mapped to [-0.5, 0.5).
__device__ __forceinline__ double splitmix_uniform(uint64_t seed, uint64_t i) {
  uint64_t z = seed + (i + 1) * 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  z = z ^ (z >> 31);
  return (double)(z >> 11) * (1.0 / 9007199254740992.0) - 0.5;
}
constexpr int kLzMax = 80;       // steps of a run, at most (and one)
constexpr int kLzThreads = 512;  // as the trial loop: one block per SM
constexpr int kLzFull = 1024;    // up to this size every step is orthogonalised in full
// Loss of orthogonality at which a step is orthogonalised (the tridiagonal
// matrix differs from that of exact arithmetic by its square).
constexpr double kLzOmega = 1e-10;

// Coefficients and recurrences of the two runs: every block forms its own copy, all
// the same, from the block partials.
struct LzState {
  double al[2][kLzMax], be[2][kLzMax], om[2][3][kLzMax + 2];  // om: rows j - 1, j, j + 1 by j mod 3
  int used[2], active[2], force[2], doit[2], done[2];         // done[0]: both runs have ended
};
// Phases: start vectors, their norms, then for every step the product, the
// recurrence, the loss of orthogonality with the sums of the orthogonalisation,
// its subtraction, and its end.
enum : int { kLzStart, kLzNorms, kLzProduct, kLzRecur, kLzLoss, kLzSubtract, kLzEnd };

// Lanczos runs of `steps` steps on the symmetric matrix Q from the start vectors
// of the seeds first + 1 .. first + ns (1 or 2 runs): out[s][0] = steps taken, then
// the diagonal and the off-diagonal entries (kLzMax each).  V: [ns][steps + 1][n]
// basis vectors, w: [ns][n].
//
// The basis is kept semi-orthogonal by partial reorthogonalisation (H. D.
// Simon, Math. Comp. 42, 1984): the recurrence for the loss of orthogonality
// runs along with the coefficients, and a step and the next one are
// orthogonalised against the whole basis only when it passes kLzOmega.  Twice
// orthogonalising every step reads the basis 4 times a step and needs 4 n j
// FP64 multiply-adds, 8 ms at n = 300,000 for the pipe alone.  The sums that a
// step needs are formed by every block from the block partials (fixed order, the
// same in all blocks).
//
// COOP: all phases in one cooperative launch, a step is 3 grid barriers.  Else a
// launch is one phase (phase, step j0), the state goes from launch to launch
// through state[2] (read from one, written to the other, by the parity of the
// launch's number), and a phase with nothing to do returns: 5 launches a step
// without a host synchronisation, for devices without cooperative launches and
// beside other solves.  The same sums in the same order: the same results.
// Measured: see Solver::lanczos.
template <int K, bool COOP>
__global__ void __launch_bounds__(kLzThreads, 1) k_lanczos(Mat<double> Q, int first, int ns, int steps, double *V,
                                                           double *w, double *part, unsigned *bar, double *out,
                                                           LzState *state, int phase, int j0, int number) {
  constexpr int NW = kLzThreads / 32;
  __shared__ LzState S;
  __shared__ double red[NW][32], tot[2][kLzMax];
  extern __shared__ __align__(16) unsigned char slots[];
  const long long n = Q.nrows;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5, nb = gridDim.x;
  Slot<double> *buf = reinterpret_cast<Slot<double> *>(slots) + wid * kTileSlots;
  unsigned gen = COOP && t == 0 ? ld_acquire_gpu(bar + kBarGen) : 0u;
  const long long e0 = (long long)blockIdx.x * kLzThreads + t, es = (long long)nb * kLzThreads;
  const WarpItems it;
  constexpr int TR = TileIter<K>::TR;
  const long long tiles = (n + TR - 1) / TR;
  // One sum per run: block partials to part, then after a barrier totals in tot[s][0].
  auto put2 = [&](double a, double b, double *dst) {
    double v[2] = {a, b};
    const double r = warp_halve<2, false>(v);
    if ((lane & 15) == 0) red[wid][lane >> 4] = r;
    __syncthreads();
    if (t < 2) {
      double x = red[0][t];
      for (int k = 1; k < NW; ++k) x += red[k][t];
      dst[2 * blockIdx.x + t] = x;
    }
  };
  auto get2 = [&](const double *src) {
    if (wid < 2) {
      double x = 0.0;
#pragma unroll 5
      for (int b = lane; b < nb; b += 32) x += __ldcg(src + 2 * b + wid);
      x = warp_sum(x);
      if (lane == 0) tot[wid][0] = x;
    }
    __syncthreads();
  };
  double *pa = part, *pb = part + 2 * kMaxBlocks, *ph = part + 4 * kMaxBlocks;  // ph: [block][2][kLzMax]
  double a[2];
  auto start = [&] {
    if (t < 2) {
      S.used[t] = S.force[t] = S.doit[t] = S.done[t] = 0;
      S.active[t] = t < ns;
    }
    a[0] = a[1] = 0.0;
    for (int s = 0; s < ns; ++s)
      for (long long i = e0; i < n; i += es) {
        const double v = splitmix_uniform((uint64_t)(first + 1 + s), (uint64_t)i);
        w[s * n + i] = v;
        a[s] += v * v;
      }
    put2(a[0], a[1], pb);
  };
  auto norms = [&] {  // normalised start vectors
    get2(pb);
    for (int s = 0; s < ns; ++s) {
      const double f = 1.0 / sqrt(tot[s][0]);
      for (long long i = e0; i < n; i += es) V[(size_t)s * (steps + 1) * n + i] = w[s * n + i] * f;
    }
  };
  auto product = [&](int j) {  // w = Q v_j and alpha_j = w . v_j
    a[0] = a[1] = 0.0;
    for (long long tile = it.first; tile < tiles; tile += it.step) {
      const long long i = tile * TR + lane;
      const bool ok = lane < TR && i < n;
      const int rb = ok ? __ldg(Q.rp + i) : 0, re = ok ? __ldg(Q.rp + i + 1) : 0;
#pragma unroll
      for (int s = 0; s < 2; ++s)
        if (S.active[s]) {
          const double *v = V + ((size_t)s * (steps + 1) + j) * n;
          const MulLd<double> f{v};
          const double q = K == 16 ? tile_long_rows<false, double>(Q.ci, Q.val, rb, re, f)
                                   : tile_rows1<false, double>(Q.ci, Q.val, rb, re, f, buf);
          if (ok) {
            w[s * n + i] = q;
            a[s] += q * v[i];
          }
        }
    }
    put2(a[0], a[1], pa);
  };
  auto recur = [&](int j) {  // w -= alpha_j v_j + beta_{j-1} v_{j-1}
    get2(pa);
    if (t < 2 && S.active[t]) {
      S.al[t][j] = tot[t][0];
      S.used[t] = j + 1;
    }
    __syncthreads();
    a[0] = a[1] = 0.0;
    for (int s = 0; s < 2; ++s)
      if (S.active[s]) {
        const double *v = V + ((size_t)s * (steps + 1) + j) * n;
        const double aj = S.al[s][j], bj = j > 0 ? S.be[s][j - 1] : 0.0;
        for (long long i = e0; i < n; i += es) {
          double x = w[s * n + i] - aj * v[i];
          if (j > 0) x -= bj * v[i - n];
          w[s * n + i] = x;
          a[s] += x * x;
        }
      }
    put2(a[0], a[1], pb);
  };
  // Loss of orthogonality of the new vector against v_0 .. v_{j-1}, a lane each;
  // where it passes kLzOmega, h = V' w over 32 basis vectors at a time (a lane's 32
  // sums are joined by halving).  True when there is any.
  auto loss = [&](int j) {
    get2(pb);
    if (wid < 2 && S.active[wid]) {
      const int s = wid;
      const double b = sqrt(tot[s][0]), eps = 1.1102230246251565e-16;
      const double *oj = S.om[s][j % 3], *om1 = S.om[s][(j + 2) % 3];
      double *on = S.om[s][(j + 1) % 3];
      double worst = 0.0;
      for (int k = lane; k < j; k += 32) {
        double x = S.be[s][k] * (k + 1 == j ? 1.0 : oj[k + 1]) + (S.al[s][k] - S.al[s][j]) * oj[k];
        if (k > 0) x += S.be[s][k - 1] * oj[k - 1];
        x -= S.be[s][j - 1] * (k + 1 == j ? 1.0 : om1[k]);
        x = (x + copysign(eps * (S.be[s][k] + b), x)) / b;
        on[k] = x;
        worst = fmax(worst, fabs(x));
      }
      worst = warp_max(worst);
      if (lane == 0) {
        on[j] = eps * sqrt((double)n);
        S.doit[s] = n <= kLzFull || S.force[s] || !(worst < kLzOmega);
        S.force[s] = S.doit[s] && !S.force[s];
        S.be[s][j] = b;
      }
    } else if (wid < 2 && lane == 0) {
      S.doit[wid] = 0;
    }
    __syncthreads();
    for (int s = 0; s < 2; ++s)
      if (S.doit[s])
        for (int p0 = 0; p0 <= j; p0 += 32) {
          double acc[32];
#pragma unroll
          for (int p = 0; p < 32; ++p) acc[p] = 0.0;
          const double *v = V + ((size_t)s * (steps + 1) + p0) * n;
          for (long long i = e0; i < n; i += es) {
            const double x = w[s * n + i];
#pragma unroll
            for (int p = 0; p < 32; ++p)
              if (p0 + p <= j) acc[p] += v[(size_t)p * n + i] * x;
          }
          const double r = warp_halve<32, false>(acc);
          red[wid][lane] = r;
          __syncthreads();
          if (t < 32) {
            double x = red[0][t];
            for (int k = 1; k < NW; ++k) x += red[k][t];
            if (p0 + t < kLzMax) ph[((size_t)blockIdx.x * 2 + s) * kLzMax + p0 + t] = x;
          }
          __syncthreads();
        }
    return (S.doit[0] | S.doit[1]) != 0;
  };
  auto subtract = [&](int j) {  // w -= V h
    for (int s = 0; s < 2; ++s)
      if (S.doit[s])
        for (int p = t; p <= j; p += kLzThreads) {
          double x = 0.0;
          for (int b = 0; b < nb; ++b) x += __ldcg(ph + ((size_t)b * 2 + s) * kLzMax + p);
          tot[s][p] = x;
        }
    __syncthreads();
    a[0] = a[1] = 0.0;
    for (int s = 0; s < 2; ++s)
      if (S.doit[s]) {
        const double *v = V + (size_t)s * (steps + 1) * n;
        for (long long i = e0; i < n; i += es) {
          double x = w[s * n + i];
          for (int p = 0; p <= j; ++p) x -= tot[s][p] * v[(size_t)p * n + i];
          w[s * n + i] = x;
          a[s] += x * x;
        }
      }
    __syncthreads();
    put2(a[0], a[1], pa);
  };
  auto ended = [&](int j) {  // the norm and the orthogonality after the subtraction
    get2(pa);
    if (t < 2 && S.doit[t]) S.be[t][j] = sqrt(tot[t][0]);
    for (int s = 0; s < 2; ++s)
      if (S.doit[s])
        for (int k = t; k < j; k += kLzThreads) S.om[s][(j + 1) % 3][k] = 1.1102230246251565e-16;
    __syncthreads();
  };
  auto next = [&](int j) {  // v_{j+1}; false (and the coefficients in out) when the runs have ended
    if (t < 2 && S.active[t]) {
      const double b = S.be[t][j];
      if (b <= 1e-12 * (fabs(S.al[t][j]) + (j > 0 ? S.be[t][j - 1] : 0.0) + 1e-300)) S.active[t] = 0;
    }
    __syncthreads();
    if (j == steps - 1 || !(S.active[0] | S.active[1])) {
      if (blockIdx.x == 0 && t < ns) {
        double *o = out + t * (2 * kLzMax + 1);
        o[0] = S.used[t];
        for (int k = 0; k < S.used[t]; ++k) {
          o[1 + k] = S.al[t][k];
          o[1 + kLzMax + k] = S.be[t][k];
        }
      }
      return false;
    }
    for (int s = 0; s < 2; ++s)
      if (S.active[s]) {
        const double f = 1.0 / S.be[s][j];
        double *v = V + ((size_t)s * (steps + 1) + j + 1) * n;
        for (long long i = e0; i < n; i += es) v[i] = w[s * n + i] * f;
      }
    return true;
  };
  if (COOP) {
    auto sync = [&] { return loop_sync<false>(bar, gen) >= 0; };
    start();
    if (!sync()) return;
    norms();
    if (!sync()) return;
    for (int j = 0; j < steps; ++j) {
      product(j);
      if (!sync()) return;
      recur(j);
      if (!sync()) return;
      if (loss(j)) {
        if (!sync()) return;
        subtract(j);
        if (!sync()) return;
        ended(j);
      }
      if (!next(j)) return;
      if (!sync()) return;
    }
  } else {
    constexpr int words = sizeof(LzState) / 4;
    int *const mine = reinterpret_cast<int *>(&S);
    if (phase != kLzStart) {
      const int *src = reinterpret_cast<const int *>(state + (number & 1));
      for (int i = t; i < words; i += kLzThreads) mine[i] = src[i];
    }
    __syncthreads();
    bool more = true;
    if (phase == kLzStart) {
      start();
    } else if (phase == kLzNorms) {
      norms();
    } else if (!S.done[0]) {
      const bool any = (S.doit[0] | S.doit[1]) != 0;
      __syncthreads();  // read before loss() sets them
      if (phase == kLzProduct) {
        product(j0);
      } else if (phase == kLzRecur) {
        recur(j0);
      } else if (phase == kLzLoss) {
        if (!loss(j0)) more = next(j0);
      } else if (any && phase == kLzSubtract) {
        subtract(j0);
      } else if (any) {
        ended(j0);
        more = next(j0);
      }
    }
    __syncthreads();
    if (t == 0 && !more) S.done[0] = 1;
    __syncthreads();
    if (blockIdx.x == 0)
      for (int i = t; i < words; i += kLzThreads) reinterpret_cast<int *>(state + ((number + 1) & 1))[i] = mine[i];
  }
}

// ---------------------------------------------------------------------------
// Initial point and penalties (Sec. 3.2.1).
// ---------------------------------------------------------------------------
// x = P_[lx,ux](x0 / Dx) (x0 already in the original coordinates, or null).
__global__ void k_init_x(long long n, const double *x0, const double *Dx, const double *lx, const double *ux,
                         double *x64, double *z) {
  PDNQP_GRID_STRIDE(i, n) {
    double v = x0 ? x0[i] / Dx[i] : 0.0;
    v = v < lx[i] ? lx[i] : v;
    v = v > ux[i] ? ux[i] : v;
    x64[i] = v;
    z[i] = v;
  }
}

// lambda (scaled) = c_s lambda0 / Dc (internal row order), inner y = -lambda.
__global__ void k_init_lambda(long long m, double *lam, const double *lam0_int, const double *Dc, double cs,
                              double *y64) {
  PDNQP_GRID_STRIDE(j, m) {
    const double l = lam0_int ? cs * lam0_int[j] / Dc[j] : 0.0;
    lam[j] = l;
    y64[j] = -l;
  }
}

// Rows of the initial point: partial sum of dist(Ax, [lc, uc])^2, and the
// residual r = A x - P(A x + lambda / sigma) once sigma is known (pass 2).
template <typename T, int G>
__global__ void __launch_bounds__(kBlock) k_init_rows(Dev<T> d, Mat<double> Ad, const double *lc, const double *uc,
                                                      double *lam, const double *sig, double *rprev, int pass) {
  const double *__restrict__ x = d.xb;
  double acc = 0.0;
  TileIter<G> ti;
  for (long long tile = ti.first; tile < d.m; tile += ti.step) {
    long long j;
    const bool own = ti.row(tile, d.m, j);
    const double ax = tile_row_sum<G, double>(Ad.rp, Ad.ci, Ad.val, tile, d.m, MulLdg<double>{x});
    if (own) {
      const double lo = lc[j], hi = uc[j];
      if (pass == 0) {
        double p = ax;
        p = p < lo ? lo : p;
        p = p > hi ? hi : p;
        acc += (ax - p) * (ax - p);
      } else {
        double s;
        if (j < d.mE) {
          s = lo;
        } else {
          s = ax + lam[j] / sig[j];
          s = s < lo ? lo : s;
          s = s > hi ? hi : s;
        }
        rprev[j] = ax - s;
      }
    }
  }
  double v[1] = {acc};
  block_reduce_store<1, 0u>(v, d.part);
}

// Partials of x'Qx (from H x - gamma^-1 x) and c'x.
template <typename T, int G>
__global__ void __launch_bounds__(kBlock) k_objective(Dev<T> d, Mat<double> Hd, const double *c, double ginv) {
  const double *__restrict__ x = d.xb;
  double xqx = 0.0, cx = 0.0;
  TileIter<G> ti;
  for (long long tile = ti.first; tile < d.n; tile += ti.step) {
    long long i;
    const bool own = ti.row(tile, d.n, i);
    const double hx = tile_row_sum<G, double>(Hd.rp, Hd.ci, Hd.val, tile, d.n, MulLdg<double>{x});
    if (own) {
      const double xi = double(x[i]);
      xqx += xi * (hx - ginv * xi);
      cx += c[i] * xi;
    }
  }
  double v[2] = {xqx, cx};
  block_reduce_store<2, 0u>(v, d.part);
}

// ---------------------------------------------------------------------------
// Outer glue (Algorithm 3).
// ---------------------------------------------------------------------------
// Quantities of the outer residual reduction:
//   0 r_p scaled, 1 s_p scaled, 2 r_p unscaled, 3 s_p unscaled, 4 ||r||_inf (rows)
//   5 r_d scaled, 6 s_d scaled, 7 r_d unscaled, 8 s_d unscaled, 9 ||x - z||_inf,
//   10 x'Qx, 11 c'x                         (10, 11 sums; the rest maxima)
// and of the infeasibility tests (Sec. "Infeasibility detection") on the scaled
// problem, from the changes over one outer iteration dlam = lambda^{k+1} -
// lambda^k and dx = x^{k+1} - x^k (unnormalised; the host divides by the norms).
// Rows (4): 0 largest |dlam_j| that would need an infinite row bound (sign
// condition), 1 sum of the finite-bound terms of sigma_C(dlam), 2 largest
// departure of (A dx)_j from the recession cone of [l_c, u_c], 3 ||dlam||_inf.
// Columns (7): 0 largest |v_i|, v = -A' dlam, that would need an infinite
// variable bound, 1 sum of the finite-bound terms of sigma_X(v), 2 largest
// departure of dx_i from the recession cone of [l_x, u_x], 3 dx'Q dx, 4 c'dx,
// 5 ||Q dx||_inf, 6 ||dx||_inf (Q dx = H dx - dx / gamma).
// Both in one pass over each matrix: the second product of a tile finds its
// entries in the caches (separate passes, each with its own reduction, read and
// synchronisation, took 0.55 ms at n = 1e6 and 0.1 ms of launches and waits at
// any size).
constexpr int OUT_Q = 12, INF_R = 4, INF_C = 7, INF_Q = INF_R + INF_C;
constexpr unsigned OUT_MAXMASK = 0x3FFu, INF_R_MAXMASK = 0xDu, INF_C_MAXMASK = 0x65u;
constexpr int kOutRows = OUT_Q + INF_R, kOutCols = OUT_Q + INF_C;  // rows of part: rows first, then columns
constexpr unsigned kOutRowsMask = OUT_MAXMASK | INF_R_MAXMASK << OUT_Q, kOutColsMask = OUT_MAXMASK | INF_C_MAXMASK << OUT_Q;
static_assert(kOutRows + kOutCols <= kMaxPartials, "partials of the outer pass");

// Terms of the termination-test maxima (Eqs. outer-residuals / outer-scales): a
// residual term that is not finite counts as +inf (a point with NaN or infinite
// entries never passes), and a scale term that is not finite is left out (an
// infinite scale would excuse any residual).
__device__ __forceinline__ double res_of(double v) { return nonfinite(v) ? INFINITY : fabs(v); }
__device__ __forceinline__ double scale_of(double v) { return nonfinite(v) ? 0.0 : fabs(v); }

// Eq. practical-multiplier-update (two-sided rows) + row terms of the residuals;
// with update also lam0 = the previous multipliers and the infeasibility terms.
template <typename T, int G>
__global__ void __launch_bounds__(kBlock) k_outer_rows(Dev<T> d, Mat<double> Ad, const double *lc, const double *uc,
                                                       const double *Dc, double *lam, double *lam0, const double *sig,
                                                       double *rcur, const double *dx, int update) {
  const double *__restrict__ x = d.xb;  // outer x (FP64)
  double q[kOutRows];
#pragma unroll
  for (int k = 0; k < kOutRows; ++k) q[k] = 0.0;
  TileIter<G> ti;
  for (long long tile = ti.first; tile < d.m; tile += ti.step) {
    const double ax = update ? tile_row_sum<G, double>(Ad.rp, Ad.ci, Ad.val, tile, d.m, MulLdg<double, sizeof(T) == 8 ? 2 : 0>{x})
                             : tile_row_sum<G, double>(Ad.rp, Ad.ci, Ad.val, tile, d.m, MulLdg<double>{x});
    const double ad =
        update ? tile_row_sum<G, double>(Ad.rp, Ad.ci, Ad.val, tile, d.m, MulLdg<double>{dx}) : 0.0;
    long long j;
    const bool own = ti.row(tile, d.m, j);
    if (own) {
      const double lo = lc[j], hi = uc[j];
      if (update) {
        const double l0 = lam[j];
        double s;
        if (j < d.mE) {
          s = lo;
        } else {
          s = clampv<double>(ax + l0 / sig[j], lo, hi);
        }
        const double r = ax - s, l1 = l0 + sig[j] * r;
        lam0[j] = l0;
        lam[j] = l1;
        rcur[j] = r;
        q[4] = max_abs(q[4], r);
        const double y = l1 - l0;
        if (y > 0.0) {
          if (isinf(hi)) q[OUT_Q] = max_abs(q[OUT_Q], y); else q[OUT_Q + 1] += hi * y;
        } else if (y < 0.0) {
          if (isinf(lo)) q[OUT_Q] = max_abs(q[OUT_Q], y); else q[OUT_Q + 1] += lo * y;
        }
        if (!isinf(lo) && ad < 0.0) q[OUT_Q + 2] = max_abs(q[OUT_Q + 2], ad);
        if (!isinf(hi) && ad > 0.0) q[OUT_Q + 2] = max_abs(q[OUT_Q + 2], ad);
        q[OUT_Q + 3] = max_abs(q[OUT_Q + 3], y);
      }
      const double viol = less_bits(ax, lo) ? lo - ax : (less_bits(hi, ax) ? ax - hi : 0.0);
      double spv = scale_of(ax);
      spv = max_abs(spv, scale_of(lo));
      spv = max_abs(spv, scale_of(hi));
      q[0] = max_abs(q[0], res_of(viol));
      q[1] = max_abs(q[1], spv);
      const double dc = Dc[j];  // divisions: these are reported, and decide termination
      q[2] = max_abs(q[2], res_of(viol / dc));
      q[3] = max_abs(q[3], spv / dc);
    }
  }
  block_reduce_store<kOutRows, kOutRowsMask>(q, d.part);
}

// Column terms: Qx = H x - gamma^-1 x, A' lambda, projected stationarity in the
// scaled and the original coordinates (x = Dx xbar, lambda = Dc lambdabar /
// c_s).  The last block joins the row and column partials into out.
template <typename T, int G>
__global__ void __launch_bounds__(kBlock) k_outer_cols(Dev<T> d, Mat<double> Hd, Mat<double> Atd, const double *c,
                                                       const double *lx, const double *ux, const double *Dx,
                                                       const double *lam, const double *lam0, const double *dx,
                                                       const double *z, double ginv, double cs, int update, int nb_r,
                                                       double *out) {
  const double *__restrict__ x = d.xb;  // outer x (FP64)
  double q[kOutCols];
#pragma unroll
  for (int k = 0; k < kOutCols; ++k) q[k] = 0.0;
  TileIter<G> ti;
  for (long long tile = ti.first; tile < d.n; tile += ti.step) {
    const double hx = tile_row_sum<G, double>(Hd.rp, Hd.ci, Hd.val, tile, d.n, MulLdg<double>{x});
    const double atl = tile_row_sum<G, double>(Atd.rp, Atd.ci, Atd.val, tile, d.n, MulLdg<double>{lam});
    double hd = 0.0, atd = 0.0;
    if (update) {
      hd = tile_row_sum<G, double>(Hd.rp, Hd.ci, Hd.val, tile, d.n, MulLdg<double>{dx});
      atd = tile_row_sum<G, double>(Atd.rp, Atd.ci, Atd.val, tile, d.n,
                                    entry([&](int k) { return lam[k] - lam0[k]; }, AddProduct()));
    }
    long long i;
    const bool own = ti.row(tile, d.n, i);
    if (own) {
      const double xi = x[i], ci = c[i], lo = lx[i], hi = ux[i], dxi = Dx[i];
      const double qx = hx - ginv * xi;
      const double g = qx + ci + atl;
      q[5] = max_abs(q[5], res_of(xi - clampv<double>(xi - g, lo, hi)));
      const double sc = max_abs(max_abs(scale_of(qx), ci), scale_of(atl));
      q[6] = max_abs(q[6], sc);
      const double f = 1.0 / (cs * dxi);
      const double xo = dxi * xi, loo = lo * dxi, hio = hi * dxi, go = g * f;
      q[7] = max_abs(q[7], res_of(xo - clampv<double>(xo - go, loo, hio)));
      q[2] = max_abs(q[2], res_of(less_bits(xo, loo) ? loo - xo : (less_bits(hio, xo) ? xo - hio : 0.0)));
      q[8] = max_abs(q[8], sc * f);
      q[9] = max_abs(q[9], xi - z[i]);
      q[10] += xi * qx;
      q[11] += ci * xi;
      if (update) {
        const double v = -atd, di = dx[i], qd = hd - ginv * di;
        double *p = q + OUT_Q;
        if (v > 0.0) {
          if (isinf(hi)) p[0] = max_abs(p[0], v); else p[1] += hi * v;
        } else if (v < 0.0) {
          if (isinf(lo)) p[0] = max_abs(p[0], v); else p[1] += lo * v;
        }
        if (!isinf(lo) && di < 0.0) p[2] = max_abs(p[2], di);
        if (!isinf(hi) && di > 0.0) p[2] = max_abs(p[2], di);
        p[3] += di * qd;
        p[4] += ci * di;
        p[5] = max_abs(p[5], qd);
        p[6] = max_abs(p[6], di);
      }
    }
  }
  block_reduce_store<kOutCols, kOutColsMask>(q, d.part + kOutRows * kMaxBlocks);
  if (arrive_last(d.ctr + 3)) {
    double a[kOutRows], b[kOutCols];
    final_reduce<kOutRows>(d.part, nb_r, kOutRowsMask, a);
    final_reduce<kOutCols>(d.part + kOutRows * kMaxBlocks, gridDim.x, kOutColsMask, b);
    if (threadIdx.x == 0) {
      for (int k = 0; k < OUT_Q; ++k) out[k] = ((OUT_MAXMASK >> k) & 1u) ? fmax(a[k], b[k]) : a[k] + b[k];
      for (int k = 0; k < INF_R; ++k) out[OUT_Q + k] = a[OUT_Q + k];
      for (int k = 0; k < INF_C; ++k) out[OUT_Q + INF_R + k] = b[OUT_Q + k];
      d.ctr[3] = 0u;
    }
  }
}

// Anderson acceleration (Sec. "Anderson acceleration"): sums of one Type-II
// step over the stored pairs (U_a, G_a), a = 0..L-1 oldest first, physical
// slot (head + a) % cap, D = m + n doubles each.  With f_a = G_a - U_a,
// dF_a = f_{a+1} - f_a (a < nc = L - 1) and f_k = f_{L-1}: out rows
// a * nc + b = dF_a'dF_b, nc * nc + a = dF_a'f_k, nc * nc + nc = f_k'f_k.
template <int NC>
__global__ void __launch_bounds__(kBlock) k_aa_dots(const double *U, const double *G, int head, int cap, long long D,
                                                    double *part) {
  constexpr int NQ = NC * NC + NC + 1;
  double q[NQ];
#pragma unroll
  for (int k = 0; k < NQ; ++k) q[k] = 0.0;
  PDNQP_GRID_STRIDE(i, D) {
    double f[NC + 1];
#pragma unroll
    for (int a = 0; a <= NC; ++a) {
      const long long s = (long long)((head + a) % cap) * D;
      f[a] = G[s + i] - U[s + i];
    }
    double df[NC];
#pragma unroll
    for (int a = 0; a < NC; ++a) df[a] = f[a + 1] - f[a];
#pragma unroll
    for (int a = 0; a < NC; ++a) {
#pragma unroll
      for (int b = 0; b < NC; ++b) q[a * NC + b] += df[a] * df[b];
      q[NC * NC + a] += df[a] * f[NC];
    }
    q[NC * NC + NC] += f[NC] * f[NC];
  }
  block_reduce_store<NQ, 0u>(q, part);
}

// The extrapolated point out = G_{L-1} - sum_a gam_a (G_{a+1} - G_a) and the
// squared norm of the correction (row 0 of part).
__global__ void __launch_bounds__(kBlock) k_aa_apply(const double *G, int head, int cap, int nc, long long D,
                                                     double g0, double g1, double g2, double g3, double *out,
                                                     double *part) {
  const double gam[4] = {g0, g1, g2, g3};
  double sn[1] = {0.0};
  PDNQP_GRID_STRIDE(i, D) {
    double v = 0.0;
    for (int a = 0; a < nc; ++a) {
      const long long s0 = (long long)((head + a) % cap) * D, s1 = (long long)((head + a + 1) % cap) * D;
      v += gam[a] * (G[s1 + i] - G[s0 + i]);
    }
    out[i] = G[(long long)((head + nc) % cap) * D + i] - v;
    sn[0] += v * v;
  }
  block_reduce_store<1, 0u>(sn, part);
}

// Eq. penalty-trigger-eq with the growth rule (only when `grow`: the primal
// part of the termination test still fails).  Stores r as the previous residual.
__global__ void k_sigma_update(int m, int mE, double *sig, const double *lam, const double *rcur, double *rprev,
                               double theta, int grow, double rn, double dsig, double smax) {
  PDNQP_GRID_STRIDE(j, m) {
    const double r = rcur[j];
    const bool active = j < mE || lam[j] != 0.0;
    if (grow && active && fabs(r) > theta * fabs(rprev[j]) && rn > 0.0)
      sig[j] = fmin(smax, sig[j] * fmax(1.0, dsig * fabs(r) / rn));
    rprev[j] = r;
  }
}

// Unscaling for the result: x_orig = Dx x, lambda_orig = Dc lambda / c_s.
template <typename T>
__global__ void k_unscale(const T *x, const double *Dx, long long n, const double *lam, const double *Dc, long long m,
                          double cs, double *xo, double *lo) {
  PDNQP_GRID_STRIDE(i, n) xo[i] = Dx[i] * double(x[i]);
  PDNQP_GRID_STRIDE(j, m) lo[j] = Dc[j] * lam[j] / cs;
}

}  // namespace
}  // namespace pdq

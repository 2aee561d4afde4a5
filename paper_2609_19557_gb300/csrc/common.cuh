// Device helpers shared by the PDNQP kernels: row sums of CSR matrices by warp
// tiles, deterministic block reductions, the grid barrier, and the device-resident
// scalar state of the inner solver.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace pdq {

constexpr int kBlock = 256;        // threads per block of every vector/SpMV kernel
constexpr int kMaxBlocks = 152 * 8;  // grid cap: 8 resident 256-thread blocks on each of 152 SMs
constexpr int kMaxPartials = 48;   // quantities reduced per launch (rows of the partials array)

// Inner-solver status kept on the device (Algorithm 4 return paths).
enum InnerStatus : int {
  ST_RUNNING = 0,
  ST_CONVERGED = 1,
  ST_ITER_LIMIT = 2,
  ST_NUMERICAL_ERROR = 3,
  ST_PAUSED = 4,
  ST_IDLE = 5,
  ST_READY = 6,  // batched form: set up, waiting for the batch scheduler to let it run
};

// Scalar state of one inner solve.  Written by the host before the solve,
// updated only by single-block kernels (decide / check-final), read by all.
struct DevState {
  int status;
  int cur;             // index (0/1) of the current iterate buffers; the trial goes to 1 - cur
  int accepted;        // the last trial was accepted: the new averages are in buffer acur ^ 1
  int acur;            // index (0/1) of the committed running averages
  int check_due;       // a stopping/restart check follows this trial
  int restart_flag;    // the last check restarts the epoch
  int restart_use_avg; // ... from the averaged candidate
  int ret_avg;         // converged candidate is the average
  int ignore_conv;     // debug: never stop on the inner termination test
  int start_status;    // status the inner-solve setup ends in: ST_RUNNING, or ST_READY in the batched form
  int xcur, xtr, xsp;  // indices (0..2) of the current, trial and spare x buffers
  int spec;            // persistent loop: the next x_tr (in x[xtr]) and the averages of x are formed already
  long long t;         // accepted steps in the current epoch (N_p = N_d, Eq. pdqp-trial)
  long long t_total;   // accepted steps in this inner solve
  long long trials;    // all trials, all solves
  long long accepted_all;
  long long restarts;
  long long rej;       // consecutive rejections
  long long k_in;      // accepted-iteration limit (Table tab:parameters)
  long long pause_at;  // debug: pause after this many accepted steps (-1: never)
  long long k_chk;     // check period
  long long rej_limit;
  long long slot_left; // trials left in the current graph launch (bounds each device loop)
  double kappa;        // common step factor of the rejection rule
  double omega;        // primal weight (Eq. primal-weight-update)
  double alpha_acc;    // alpha of the last accepted trial
  double k_restart;    // restart metric at the start of the epoch
  double k_last;       // restart metric of the candidate at the previous check
  double dta, dtr;     // inner tolerances delta_a, delta_r
  double shrink;       // kappa factor on rejection
  double beta_suff, beta_nec, beta_art;
  double chk[16];      // reductions of the last check (diagnostics)
  // Scalars of the next trial, formed once where t, kappa, omega or alpha_acc
  // change, in both storage types (kAlpha ..).  Formed by every thread of every
  // pass they took 4 FP64 divisions a thread (5 us a pass with 24 warps on an
  // SM's FP64 pipe).
  double sd[12];
  float sf[12];
};

// Slots of DevState::sd / sf: alpha, 1 - alpha, beta, kappa / omega, kappa
// omega, alpha_acc, 1 - alpha_acc; alpha and 1 - alpha of the trial after an
// acceptance; omega / kappa and 1 / (kappa omega) (acceptance test, FP64 only).
enum : int { kAlpha, kOma, kBeta, kSct, kSce, kAp, kOmap, kAlpha1, kOma1, kOka, kIko };

// Scalars of one trial in the storage type T.
template <typename T>
struct Scal {
  const T *v;
  __device__ __forceinline__ explicit Scal(const DevState *st) : v(pick(st, T(0))) {}
  __device__ __forceinline__ T operator[](int k) const { return v[k]; }
  static __device__ __forceinline__ const double *pick(const DevState *st, double) { return st->sd; }
  static __device__ __forceinline__ const float *pick(const DevState *st, float) { return st->sf; }
};

__host__ __device__ inline void set_scalar(DevState *S, int k, double v) {
  S->sd[k] = v;
  S->sf[k] = (float)v;
}
// A weight and its complement (formed in the storage type).
__host__ __device__ inline void set_weight(DevState *S, int k, double v) {
  set_scalar(S, k, v);
  S->sd[k + 1] = 1.0 - v;
  S->sf[k + 1] = 1.0f - (float)v;
}
__host__ __device__ inline void refresh_scalars(DevState *S) {
  const double t = (double)S->t;
  set_weight(S, kAlpha, 2.0 / (t + 2.0));
  set_scalar(S, kBeta, t / (t + 1.0));
  set_scalar(S, kSct, S->kappa / S->omega);
  set_scalar(S, kSce, S->kappa * S->omega);
  set_weight(S, kAp, S->alpha_acc);
  set_weight(S, kAlpha1, 2.0 / (t + 3.0));
  S->sd[kOka] = S->omega / S->kappa;
  S->sd[kIko] = 1.0 / (S->kappa * S->omega);
}
// After an acceptance (t has advanced by one; kappa and omega have not
// changed): the weights move on, and only alpha of the trial after the next and
// beta are new (alpha1, beta: their values for the new t).
__host__ __device__ inline void advance_scalars(DevState *S, double alpha1, double beta) {
  for (int k = 0; k < 2; ++k) {
    S->sd[kAp + k] = S->sd[kAlpha + k];
    S->sf[kAp + k] = S->sf[kAlpha + k];
    S->sd[kAlpha + k] = S->sd[kAlpha1 + k];
    S->sf[kAlpha + k] = S->sf[kAlpha1 + k];
  }
  set_weight(S, kAlpha1, alpha1);
  set_scalar(S, kBeta, beta);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
// The blocks a kernel's work is spread over: the hardware grid, or, in the
// batched form, the contiguous run of blocks of one launch that one problem
// of the batch owns (block b of nb).  Reductions and grid-stride loops use
// it instead of blockIdx / gridDim, so a problem sees the same partition
// (and the same rounding) whether it runs alone or in a batch.
struct GridCtx {
  int b, nb;
};
__device__ __forceinline__ GridCtx hw_grid() { return GridCtx{(int)blockIdx.x, (int)gridDim.x}; }

// Tests and comparisons of doubles on the integer pipes, a few instructions
// each, instead of 16 cycles of the SM's FP64 pipe.  They work on the two words
// (from the intrinsics: on the 64-bit pattern the compiler recognises the
// floating-point test and emits it again).
typedef unsigned long long u64;
constexpr u64 kInfBits = 0x7ff0000000000000ull;
__device__ __forceinline__ u64 abs_bits(double v) {
  return ((u64)(unsigned)(__double2hiint(v) & 0x7fffffff) << 32) | (unsigned)__double2loint(v);
}
__device__ __forceinline__ bool nonfinite(double v) { return (__double2hiint(v) & 0x7fffffff) >= 0x7ff00000; }
__device__ __forceinline__ bool is_nan_bits(double v) {
  const int h = __double2hiint(v) & 0x7fffffff;
  return h > 0x7ff00000 || (h == 0x7ff00000 && __double2loint(v) != 0);
}
// Order-preserving key (-0 before +0; NaN beyond the infinity of its sign).
__device__ __forceinline__ long long order_key(double v) {
  const int h = __double2hiint(v), s = h >> 31;
  return ((long long)(h ^ (s & 0x7fffffff)) << 32) | (unsigned)(__double2loint(v) ^ s);
}
// a < b; false when either is NaN.
__device__ __forceinline__ bool less_bits(double a, double b) {
  return order_key(a) < order_key(b) && !is_nan_bits(a) && !is_nan_bits(b);
}
// Maximum of a non-negative `a` and |v|; a NaN v is left out (as fmax does).
__device__ __forceinline__ double max_abs(double a, double v) {
  const u64 b = abs_bits(v);
  return b > abs_bits(a) && !is_nan_bits(v) ? __hiloint2double((int)(b >> 32), (int)(unsigned)b) : a;
}
__device__ __forceinline__ float max_abs(float a, float v) { return fmaxf(a, fabsf(v)); }

// FP32 value as a double without the conversion instruction (which runs on the
// FP64 pipe): exact; denormals, infinities and NaN take the instruction.
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v) {
  const unsigned u = __float_as_uint(v), m = u & 0x7fffffffu;
  if (m - 0x00800000u >= 0x7f000000u && m != 0u) return double(v);
  return __hiloint2double((int)((u & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u)), (int)(u << 29));
}

// Reciprocal of a positive double by two Newton steps from the FP32 reciprocal
// (4 FP64 instructions; a division is several times that), within 0.51 units in the
// last place (a quotient formed with it: 1.5); outside FP32's range the division.
__device__ __forceinline__ double recip(double v) {
  const float f = (float)v;
  if (!(f > 1e-30f && f < 1e30f)) return 1.0 / v;
  double r = widen(1.0f / f);
  r = fma(r, fma(-v, r, 1.0), r);
  return fma(r, fma(-v, r, 1.0), r);
}
__device__ __forceinline__ double recip(float v) {
  if (!(v > 1e-30f && v < 1e30f)) return 1.0 / double(v);
  const double d = widen(v);
  double r = widen(1.0f / v);
  r = fma(r, fma(-d, r, 1.0), r);
  return fma(r, fma(-d, r, 1.0), r);
}

// Reciprocal square root in the storage precision.  FP64: two Newton steps from
// the FP32 value (8 FP64 instructions), within 1.01 units in the last place;
// outside FP32's range the library's.
__device__ __forceinline__ float rsqrt_t(float v) { return rsqrtf(v); }
__device__ __forceinline__ double rsqrt_t(double v) {
  const float f = (float)v;
  if (!(f > 1e-30f && f < 1e30f)) return rsqrt(v);
  double r = widen(rsqrtf(f));
  const double h = 0.5 * v;
  r = fma(r, fma(-h * r, r, 0.5), r);
  return fma(r, fma(-h * r, r, 0.5), r);
}

__host__ __device__ constexpr int count_bits(unsigned m) { return m == 0u ? 0 : (int)(m & 1u) + count_bits(m >> 1); }
__host__ __device__ constexpr int next_pow2(int v) {
  int p = 1;
  while (p < v) p *= 2;
  return p;
}

// Reduction of P values (a power of two up to 32) of every lane over the warp
// by halving: at each level a lane hands over half of its values and joins the
// other half, so P - 1 + log2(32 / P) additions instead of 5 P.  Lane l ends
// with value l / (32 / P).
template <int P, bool IsMax>
__device__ __forceinline__ double warp_halve(double (&v)[P]) {
  const int lane = threadIdx.x & 31;
  int w = 16;
#pragma unroll
  for (int h = P / 2; h > 0; h >>= 1, w >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int t = 0; t < h; ++t) {
      const double keep = up ? v[t + h] : v[t], give = up ? v[t] : v[t + h];
      const double o = __shfl_xor_sync(0xffffffffu, give, w);
      v[t] = IsMax ? max_abs(keep, o) : keep + o;
    }
  }
  double r = v[0];
#pragma unroll
  for (; w > 0; w >>= 1) {
    const double o = __shfl_xor_sync(0xffffffffu, r, w);
    r = IsMax ? max_abs(r, o) : r + o;
  }
  return r;
}

// Block reduction of NQ doubles; bit q of MASK: 0 sum, 1 maximum (of
// non-negative values).  The block writes part[q * kMaxBlocks + blk].  Must be
// called by every thread of the block (up to 512).  Sums and maxima are
// reduced over the warp by halving, then one thread per quantity joins the
// warps' values in order.  Fixed order: deterministic for a fixed grid.
template <int NQ, unsigned MASK>
__device__ __forceinline__ void block_reduce_store(double (&v)[NQ], double *part, int blk = -1) {
  if (blk < 0) blk = blockIdx.x;
  constexpr int NM = count_bits(MASK), NS = NQ - NM;
  constexpr int PS = next_pow2(NS > 0 ? NS : 1), PM = next_pow2(NM > 0 ? NM : 1);
  static_assert(PS <= 32 && PM <= 32, "at most 32 quantities of a kind");
  __shared__ double sm[NQ][16];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, nw = blockDim.x >> 5;
  double s[PS], m[PM];
#pragma unroll
  for (int k = 0; k < PS; ++k) s[k] = 0.0;
#pragma unroll
  for (int k = 0; k < PM; ++k) m[k] = 0.0;
  // idx: quantity of each slot (compile time after unrolling).
  int is = 0, im = 0;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    if ((MASK >> q) & 1u)
      m[im++] = v[q];
    else
      s[is++] = v[q];
  }
  __syncthreads();  // sm of an earlier call has been read
  const double rs = NS > 0 ? warp_halve<PS, false>(s) : 0.0, rm = NM > 0 ? warp_halve<PM, true>(m) : 0.0;
  is = 0;
  im = 0;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    if ((MASK >> q) & 1u) {
      if (lane == im * (32 / PM)) sm[q][w] = rm;
      ++im;
    } else {
      if (lane == is * (32 / PS)) sm[q][w] = rs;
      ++is;
    }
  }
  __syncthreads();
  if (t < NQ) {
    const bool mx = (MASK >> t) & 1u;
    double a = sm[t][0];
    for (int k = 1; k < nw; ++k) a = mx ? max_abs(a, sm[t][k]) : a + sm[t][k];
    part[t * kMaxBlocks + blk] = a;
  }
  __syncthreads();
}

// Polls of a grid barrier before it gives up (about two seconds) ...
constexpr unsigned kSpinLimit = 1u << 22;
// ... and further ones where a warp may go through a row of `longest` entries while
// the other blocks wait: in entry order (one_row) that takes 64 cycles an entry, and a
// poll, a round trip to L2, takes some 250 at least.
__host__ __device__ constexpr unsigned spin_more(long long longest) { return (unsigned)(longest / 2); }

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_gpu(unsigned *p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Device-wide nanosecond timer (phase timing of the persistent loop).
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// Word offsets of the barrier's generation and fault flag from its arrival
// counter: each on its own 128-byte line, so that the polls of the
// generation do not queue behind the arrival atomics.
constexpr int kBarGen = 32, kBarFault = 64, kBarWords = 96;
constexpr int kBarMore = kBarFault + 1;  // further polls (spin_more), read with the fault flag

// Barrier of one thread-block cluster.  A hardware wait without a limit, as
// __syncthreads is: the hardware starts the blocks of a cluster together, and
// every block takes the same branches, on the same state, up to each barrier.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}
// The barrier alone.
template <bool CLU, bool MORE = true>
__device__ __forceinline__ int loop_sync(unsigned *bar, unsigned &gen);

// Grid barrier of a cooperative (co-resident) launch, the wait of every kernel
// that spans blocks.  bar[0] counts the arrivals, bar[kBarGen] is the generation
// with a message in its low bit, bar[kBarFault] the fault flag.  The last block to
// arrive runs lead() with all its threads before it releases the others, so
// lead() sees every block's writes from before the barrier and every block sees
// lead()'s writes after it; what lead() returned (0 or 1) is the message, which
// every block gets.  The arrivals are reset before lead() runs, and `gen` is the
// caller's copy of the generation (thread 0), so a waiting block polls one word
// and, every 64 polls, the fault flag (each is a round trip to L2) and the words
// beside it.
//
// The wait is bounded: a block that polls kSpinLimit times (MORE: and bar[kBarMore])
// without a release, or that sees the fault flag, sets the flag and gets -1; the
// caller then leaves the kernel, so a barrier that can never complete ends the launch
// instead of hanging it.  The trial loop does without MORE: its warps take a row 256
// entries a round, so that kSpinLimit covers some 10^8 of them, and a limit that is
// not a constant costs its row pass 0.5 us of 24 (n = 1e6, FP32).
//
// CLU: the grid is one thread-block cluster (small problems), whose hardware
// barrier orders the blocks' memory accesses like a block barrier (about 0.3 us
// where the grid barrier takes 1.5 to 2.5); block 0 runs lead(), and no message
// comes back.
template <bool CLU, bool MORE = true, typename F>
__device__ __forceinline__ int loop_sync(unsigned *bar, unsigned &gen, F lead) {
  __shared__ int role;  // message, -1 fault, 2 leader
  __syncthreads();
  if (gridDim.x == 1) {
    const int msg = lead();
    __syncthreads();
    return msg;
  }
  if (CLU) {
    cluster_sync();
    if (blockIdx.x == 0) lead();
    cluster_sync();
    return 0;
  }
  if (threadIdx.x == 0) {
    __threadfence();
    role = -2;
    if (atomicAdd(bar, 1u) == gridDim.x - 1) {
      atomicExch(bar, 0u);
      __threadfence();
      role = 2;
    } else {
      unsigned it = 0, v;
      while ((v = ld_acquire_gpu(bar + kBarGen)) == gen) {
        ++it;
        const bool look = (it & 63u) == 0u;
        if (MORE ? look && (ld_acquire_gpu(bar + kBarFault) != 0u || it > kSpinLimit + ld_acquire_gpu(bar + kBarMore))
                 : it > kSpinLimit || (look && ld_acquire_gpu(bar + kBarFault) != 0u)) {
          atomicExch(bar + kBarFault, 1u);
          role = -1;
          break;
        }
      }
      if (role != -1) {
        gen = v;
        role = (int)(v & 1u);
      }
    }
  }
  __syncthreads();
  if (role != 2) return role;
  const int msg = lead();
  __syncthreads();
  if (threadIdx.x == 0) {
    gen = ((gen >> 1) + 1u) << 1 | (unsigned)msg;
    __threadfence();
    st_release_gpu(bar + kBarGen, gen);
  }
  return msg;
}

template <bool CLU, bool MORE>
__device__ __forceinline__ int loop_sync(unsigned *bar, unsigned &gen) {
  if (CLU && gridDim.x > 1) {
    cluster_sync();
    return 0;
  }
  return loop_sync<CLU, MORE>(bar, gen, [] { return 0; });
}

// Single-block final reduction of NQ quantities over nb partials (fixed order):
// warp w handles quantities w, w + nwarps, ...; lane l sums partials l, l + 32,
// ... serially, then a fixed butterfly combines the 32 lane sums.  Every thread
// of the block gets out[].  blockDim.x must be a multiple of 32.
template <int NQ>
__device__ __forceinline__ void final_reduce(const double *part, int nb, const unsigned kind_mask, double (&out)[NQ]) {
  __shared__ double res[NQ];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int q = wid; q < NQ; q += nw) {
    const bool mx = (kind_mask >> q) & 1u;
    double a = 0.0;
    for (int b = lane; b < nb; b += 32) {
      const double p = __ldcg(part + q * kMaxBlocks + b);
      a = mx ? fmax(a, p) : a + p;
    }
    a = mx ? warp_max(a) : warp_sum(a);  // fixed butterfly: deterministic
    if (lane == 0) res[q] = a;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NQ; ++q) out[q] = res[q];
  __syncthreads();
}

// Warp tiles of consecutive rows: lane l < TR owns row tile + l (coalesced
// per-row loads and stores).  K: lane setting of the matrix the kernel works
// through (tile_reduce): 32 rows a warp, 8 with K = 16, where a row keeps the
// whole warp busy (on rows of 100 entries, 8 x 32 entries are in flight either
// way, and a small matrix spreads over four times as many warps).
template <int K>
struct TileIter {
  static constexpr int TR = K == 16 ? 8 : 32;
  int lane;
  long long first, step;
  __device__ __forceinline__ TileIter(GridCtx g = hw_grid()) {
    lane = threadIdx.x & 31;
    first = ((long long)(threadIdx.x >> 5) * g.nb + g.b) * TR;  // a few tiles spread over all blocks
    step = (((long long)g.nb * blockDim.x) >> 5) * TR;
  }
  // Row of this lane in a tile; false past the tile or the matrix.
  __device__ __forceinline__ bool row(long long tile, long long nrows, long long &i) const {
    i = tile + lane;
    return (TR == 32 || lane < TR) && i < nrows;
  }
};
// Rows one block of a tile kernel takes in a trip.
inline int tile_rows_per_block(int k) { return kBlock / 32 * (k == 16 ? 8 : 32); }

// ---------------------------------------------------------------------------
// Row reductions of CSR matrices, one warp per tile of consecutive rows.  Lane
// l brings the entry range [rb, re) of row tile + l (empty past the matrix)
// and gets that row's sum (or maximum): F::gather(col) loads what an entry
// multiplies, F::add(acc, val, x) adds the entry.  The order of every sum is
// fixed.  A round looks up to 512 entries past the end of its row, beyond 2^31 - 1
// in the last rows of the largest matrices: positions are unsigned, or what is
// compared is the entries left in the row (end - position, as a signed number; in
// tile_rows that takes registers which the FP32 column pass does not have: 57.5 ms
// a call at n = 1e6 instead of 54.8).
//
// What the two forms are built around: gathers are bound by memory latency, so
// a warp issues the 8 index and value loads of a round, then the 8 gathers (16
// with two matrices) before it uses any; and an FP64 instruction occupies its
// SM's pipe for 16 cycles however many lanes are active, so no step may run
// with few of them.
// ---------------------------------------------------------------------------
template <typename Acc>
struct __align__(2 * sizeof(Acc)) Slot {
  Acc a, x;
};
constexpr int kSlotLd = 9;                     // slots of a row in a round's buffer (8 and one of padding)
constexpr int kTileSlots = 32 * kSlotLd;       // slots of one warp
constexpr int kLongRowEntries = 32;            // longer rows are summed by the whole warp
constexpr int kDenseRow = 1024;                // see one_row
constexpr int kRowAlone = 512;                 // rows this long get a warp's 256 entries a round (tile_long_rows gives a row 32)

template <bool IsMax, typename A>
__device__ __forceinline__ A acc_join(A a, A b) {  // maxima: of non-negative values
  return IsMax ? max_abs(a, b) : a + b;
}

// One row of any length by the whole warp, 256 entries a round; every lane
// gets the result.
template <bool IsMax, typename Acc, typename T, typename F>
__device__ __forceinline__ Acc warp_row(const int *__restrict__ ci, const T *__restrict__ val, int b, int e,
                                        const F &f) {
  const int lane = threadIdx.x & 31;
  Acc acc = Acc(0);
  for (unsigned k0 = (unsigned)b + lane;; k0 += 256) {
    const int left = (int)((unsigned)e - k0);
    if (left + lane <= 0) break;  // the same for the whole warp
    int c[8];
    T a[8];
    Acc p[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const bool ok = left > 32 * u;
      c[u] = ok ? __ldg(ci + k0 + 32 * u) : -1;
      a[u] = ok ? __ldg(val + k0 + 32 * u) : T(0);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) p[u] = c[u] >= 0 ? f.gather(c[u]) : Acc(0);
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (left + lane > 32 * u) {  // the same for the whole warp
        if (c[u] >= 0) f.add(acc, Acc(a[u]), p[u]);
      }
  }
#pragma unroll
  for (int w = 16; w > 0; w >>= 1) acc = acc_join<IsMax>(acc, __shfl_xor_sync(0xffffffffu, acc, w));
  return acc;
}

// The buffer of tile_rows for one warp and one matrix (kernels of kBlock
// threads; FP32 needs none).
template <typename Acc>
__device__ __forceinline__ Slot<Acc> *warp_slots() {
  if (sizeof(Acc) == 4) return nullptr;
  __shared__ Slot<double> buf[kBlock / 32][kTileSlots];
  return reinterpret_cast<Slot<Acc> *>(buf[threadIdx.x >> 5]);
}

// A row by one warp, in the order F asks for.  kOrder = 1 or 2: a dense row (more
// than kDenseRow entries) is added entry by entry from the first, each with a
// multiply-add (1) or its product rounded first (2).  The residual of a dense
// equality row (the simplex row of a Motzkin-Straus problem) is a difference of
// nearly equal numbers, and its multiplier follows the rounding of that sum: in
// another order it moves by some 1e-9 of itself at 10,000 entries, so the two
// kernels that take it (base point, multiplier update: once an outer iteration)
// keep the order they always had (buf: the warp's slots).  Operands are loaded and gathered 256 at a
// time; what is left is the chain of additions, 64 cycles each (0.3 ms at
// 10,000 entries).
template <bool IsMax, typename Acc, typename T, typename F>
__device__ __forceinline__ Acc one_row(const int *__restrict__ ci, const T *__restrict__ val, int b, int e, const F &f,
                                       Slot<Acc> *buf) {
  if constexpr (F::kOrder == 0) {
    return warp_row<IsMax, Acc>(ci, val, b, e, f);
  } else {
    if (e - b <= kDenseRow) return warp_row<IsMax, Acc>(ci, val, b, e, f);
    const int lane = threadIdx.x & 31;
    Acc acc = Acc(0);
    for (unsigned k0 = b; k0 < (unsigned)e; k0 += 256) {
      Slot<Acc> r[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const unsigned k = k0 + 32 * u + lane;
        r[u] = k < (unsigned)e ? Slot<Acc>{Acc(__ldg(val + k)), f.gather(__ldg(ci + k))} : Slot<Acc>{Acc(0), Acc(0)};
        if (F::kOrder == 2) r[u].x = __dmul_rn(r[u].a, r[u].x);
      }
      __syncwarp();
      int cnt = 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) {  // entries that multiply zero change nothing: left out
        const unsigned nz = __ballot_sync(0xffffffffu, r[u].x != Acc(0));
        if (r[u].x != Acc(0)) buf[cnt + __popc(nz & ((1u << lane) - 1u))] = r[u];
        cnt += __popc(nz);
      }
      __syncwarp();
      int k = 0;
      for (; k + 8 <= cnt; k += 8) {
        Slot<Acc> v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = buf[k + u];
#pragma unroll
        for (int u = 0; u < 8; ++u) acc = F::kOrder == 1 ? fma(v[u].a, v[u].x, acc) : acc + v[u].x;
      }
      for (; k < cnt; ++k) acc = F::kOrder == 1 ? fma(buf[k].a, buf[k].x, acc) : acc + buf[k].x;
    }
    __syncwarp();
    return acc;
  }
}

// Short rows (32 of them, NM matrices with the same rows).  A round takes 8
// entries of every row: groups of 4 lanes load them (two steps of 8 rows x 4
// entries per quarter of the tile, so the loads of a step are consecutive in
// memory) and gather.
//   FP64: value and operand go to the warp's buffer, from which lane l adds its
// own row's entries in order, one multiply-add each: per round and matrix at
// most 8 FP64 steps, all with the rows that still have entries, where sums
// across lanes would add idle lanes and a reduction.
//   FP32: the lanes add their entries, and the 4 partial sums of a row are
// joined by halving (3 additions and 4 shuffles for the 32 rows): arithmetic is
// cheap, and the buffer would cost 16 shared-memory accesses a round.
// Rows of more than kLongRowEntries entries are left out of the rounds and
// summed by warp_row, so that one of them does not hold up its tile.  buf:
// kTileSlots slots of this warp (FP32: unused).  LongRows = false: the caller
// has taken the long rows out.  The matrices take turns in the slots: a set for
// each would take 147 KB of a block of 16 warps' L1, one set 74 KB.
template <int NM, bool IsMax, typename Acc, bool LongRows = true, typename T, typename F>
__device__ __forceinline__ void tile_rows(const int *const (&ci)[NM], const T *const (&val)[NM], const int (&rb)[NM],
                                          const int (&re)[NM], const F (&f)[NM], Slot<Acc> *buf, Acc (&out)[NM]) {
  const int lane = threadIdx.x & 31, sub = lane >> 2, lg = lane & 3;
  int se[NM], most = 0;
  bool lng = false;
#pragma unroll
  for (int m = 0; m < NM; ++m) {
    const bool l = LongRows && re[m] - rb[m] > kLongRowEntries;
    lng |= l;
    se[m] = l ? rb[m] : re[m];
    most = max(most, se[m] - rb[m]);
    out[m] = Acc(0);
  }
  const int longest = (int)__reduce_max_sync(0xffffffffu, (unsigned)most);
  constexpr bool kHalve = sizeof(Acc) == 4;
  Acc part[NM][4];
#pragma unroll
  for (int m = 0; m < NM; ++m)
#pragma unroll
    for (int t = 0; t < 4; ++t) part[m][t] = Acc(0);
  for (int s = 0; s < longest; s += 8) {
    int c[NM][4][2];
    T a[NM][4][2];
#pragma unroll
    for (int m = 0; m < NM; ++m)
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const unsigned p = (unsigned)__shfl_sync(0xffffffffu, rb[m], t * 8 + sub) + s + lg;
        const unsigned e = __shfl_sync(0xffffffffu, se[m], t * 8 + sub);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const bool ok = p + 4 * u < e;
          c[m][t][u] = ok ? __ldg(ci[m] + p + 4 * u) : -1;
          a[m][t][u] = ok ? __ldg(val[m] + p + 4 * u) : T(0);
        }
      }
    Acc x[NM][4][2];
#pragma unroll
    for (int m = 0; m < NM; ++m)
#pragma unroll
      for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int u = 0; u < 2; ++u) x[m][t][u] = c[m][t][u] >= 0 ? f[m].gather(c[m][t][u]) : Acc(0);
    if (kHalve) {
#pragma unroll
      for (int m = 0; m < NM; ++m)
#pragma unroll
        for (int t = 0; t < 4; ++t)
#pragma unroll
          for (int u = 0; u < 2; ++u)
            if (c[m][t][u] >= 0) f[m].add(part[m][t], Acc(a[m][t][u]), x[m][t][u]);
      continue;
    }
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      __syncwarp();  // the slots written last have been read
#pragma unroll
      for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int u = 0; u < 2; ++u)
          if (c[m][t][u] >= 0)
            buf[(t * 8 + sub) * kSlotLd + 4 * u + lg] = Slot<Acc>{Acc(a[m][t][u]), x[m][t][u]};
      __syncwarp();
      const int n = se[m] - rb[m] - s;
      const Slot<Acc> *row = buf + lane * kSlotLd;
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (j < longest - s) {  // the same for the whole warp
          if (j < n) f[m].add(out[m], row[j].a, row[j].x);
        }
    }
  }
  if (kHalve) {
    // Lane lg of a group keeps quarter lg: hands over two quarters, then one.
    const bool u2 = (lg & 2) != 0, u1 = (lg & 1) != 0;
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      Acc v[2];
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const Acc keep = u2 ? part[m][t + 2] : part[m][t], give = u2 ? part[m][t] : part[m][t + 2];
        v[t] = acc_join<IsMax>(keep, __shfl_xor_sync(0xffffffffu, give, 2));
      }
      const Acc keep = u1 ? v[1] : v[0], give = u1 ? v[0] : v[1];
      const Acc r = acc_join<IsMax>(keep, __shfl_xor_sync(0xffffffffu, give, 1));
      out[m] = __shfl_sync(0xffffffffu, r, (lane & 7) * 4 + (lane >> 3));  // row 8 lg + sub
    }
  }
  unsigned todo = LongRows ? __ballot_sync(0xffffffffu, lng) : 0u;
  while (todo) {
    const int l = __ffs(todo) - 1;
    todo &= todo - 1;
#pragma unroll
    for (int m = 0; m < NM; ++m) {
      const int b = __shfl_sync(0xffffffffu, rb[m], l), e = __shfl_sync(0xffffffffu, re[m], l);
      if (e - b > kLongRowEntries) {
        const Acc v = one_row<IsMax, Acc>(ci[m], val[m], b, e, f[m], buf);
        if (lane == l) out[m] = v;
      }
    }
  }
  __syncwarp();  // the slots may be written again
}

// One matrix.
template <bool IsMax, typename Acc, bool LongRows = true, typename T, typename F>
__device__ __forceinline__ Acc tile_rows1(const int *ci, const T *val, int rb, int re, const F &f, Slot<Acc> *buf) {
  const int *const ca[1] = {ci};
  const T *const va[1] = {val};
  const int ba[1] = {rb}, ea[1] = {re};
  const F fa[1] = {f};
  Acc out[1];
  tile_rows<1, IsMax, Acc, LongRows>(ca, va, ba, ea, fa, buf, out);
  return out[0];
}

// Long rows (8 of them, brought by lanes 0..7; lane l gets row l mod 8): all 32 lanes on each row, the 8 rows
// together (a round takes 32 entries of each).  The lanes' partial sums are
// reduced by halving: at every level a lane hands over half of its rows and
// adds the other half, 9 additions for the 8 rows instead of 40.
template <bool IsMax, typename Acc, typename T, typename F>
__device__ __forceinline__ Acc tile_long_rows(const int *__restrict__ ci, const T *__restrict__ val, int rb, int re,
                                              const F &f, Slot<Acc> *buf = nullptr) {
  const int lane = threadIdx.x & 31;
  const bool alone = re - rb > kRowAlone;
  const int se = alone ? rb : re;
  const int longest = (int)__reduce_max_sync(0xffffffffu, (unsigned)(se - rb));
  unsigned pos[8];
  int left[8];
  Acc acc[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    pos[t] = __shfl_sync(0xffffffffu, rb, t) + lane;
    left[t] = (int)((unsigned)__shfl_sync(0xffffffffu, se, t) - pos[t]);
    acc[t] = Acc(0);
  }
  for (int s = 0; s < longest; s += 32) {
    int c[8];
    T a[8];
    Acc p[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const bool ok = left[t] > s;
      c[t] = ok ? __ldg(ci + pos[t] + s) : -1;
      a[t] = ok ? __ldg(val + pos[t] + s) : T(0);
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) p[t] = c[t] >= 0 ? f.gather(c[t]) : Acc(0);
#pragma unroll
    for (int t = 0; t < 8; ++t)
      if (left[t] + lane > s) {  // the same for the whole warp
        if (c[t] >= 0) f.add(acc[t], Acc(a[t]), p[t]);
      }
  }
  int w = 16;
#pragma unroll
  for (int h = 4; h > 0; h >>= 1, w >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int t = 0; t < h; ++t) {
      const Acc keep = up ? acc[t + h] : acc[t], give = up ? acc[t] : acc[t + h];
      acc[t] = acc_join<IsMax>(keep, __shfl_xor_sync(0xffffffffu, give, w));
    }
  }
#pragma unroll
  for (int v = 2; v > 0; v >>= 1) acc[0] = acc_join<IsMax>(acc[0], __shfl_xor_sync(0xffffffffu, acc[0], v));
  Acc out = __shfl_sync(0xffffffffu, acc[0], (lane & 7) * 4);  // row l ended in lanes 4 l .. 4 l + 3
  unsigned todo = __ballot_sync(0xffffffffu, alone);
  while (todo) {
    const int l = __ffs(todo) - 1;
    todo &= todo - 1;
    const Acc v = one_row<IsMax, Acc>(ci, val, __shfl_sync(0xffffffffu, rb, l), __shfl_sync(0xffffffffu, re, l), f, buf);
    if ((lane & 7) == l) out = v;
  }
  return out;
}

// What an entry multiplies (gather) and how it is added (add), as two lambdas.
template <typename G, typename A>
struct Entry {
  static constexpr int kOrder = 0;
  G g;
  A a;
  template <typename I>
  __device__ __forceinline__ auto gather(I k) const { return g(k); }
  template <typename Acc>
  __device__ __forceinline__ void add(Acc &acc, Acc v, Acc x) const { a(acc, v, x); }
};
template <typename G, typename A>
__device__ __forceinline__ Entry<G, A> entry(G g, A a) {
  return Entry<G, A>{g, a};
}
// The usual ways to add an entry.
struct AddProduct {
  template <typename Acc>
  __device__ __forceinline__ void operator()(Acc &acc, Acc v, Acc x) const { acc += v * x; }
};
struct AddAbs {
  template <typename Acc>
  __device__ __forceinline__ void operator()(Acc &acc, Acc v, Acc x) const { acc += fabs(v * x); }
};
struct MaxAbs {
  template <typename Acc>
  __device__ __forceinline__ void operator()(Acc &acc, Acc v, Acc x) const { acc = max_abs(acc, v * x); }
};

// Row reduction of a warp tile (TileIter<K>); lane l gets row tile + l.  K: the
// matrix's lane setting, 16 = long rows (8 rows, all 32 lanes on each), 8 = short
// rows (32 rows).
template <int K, bool IsMax, typename Acc, typename T, typename F>
__device__ __forceinline__ Acc tile_reduce(const int *rp, const int *ci, const T *val, long long tile, long long nrows,
                                           const F &f, Slot<Acc> *buf) {
  const long long my = tile + (threadIdx.x & 31);
  const bool ok = (threadIdx.x & 31) < TileIter<K>::TR && my < nrows;
  const int rb = ok ? rp[my] : 0, re = ok ? rp[my + 1] : 0;
  return K == 16 ? tile_long_rows<IsMax, Acc>(ci, val, rb, re, f, buf)
                 : tile_rows1<IsMax, Acc>(ci, val, rb, re, f, buf);
}
template <int K, typename Acc, typename T, typename F>
__device__ __forceinline__ Acc tile_row_sum(const int *rp, const int *ci, const T *val, long long tile, long long nrows,
                                            const F &f, Slot<Acc> *buf = warp_slots<Acc>()) {
  return tile_reduce<K, false, Acc>(rp, ci, val, tile, nrows, f, buf);
}
template <int K, typename Acc, typename T, typename F>
__device__ __forceinline__ Acc tile_row_max(const int *rp, const int *ci, const T *val, long long tile, long long nrows,
                                            const F &f, Slot<Acc> *buf = warp_slots<Acc>()) {
  return tile_reduce<K, true, Acc>(rp, ci, val, tile, nrows, f, buf);
}

// Product with a vector that other blocks wrote before the last grid barrier of
// the same launch (not through the read-only path).
template <typename T>
struct MulLd {
  static constexpr int kOrder = 0;
  const T *x;
  __device__ __forceinline__ T gather(int k) const { return x[k]; }
  __device__ __forceinline__ void add(T &acc, T a, T v) const { acc += a * v; }
};

// Product with a vector that no block writes meanwhile.
template <typename T, int Order = 0>
struct MulLdg {
  static constexpr int kOrder = Order;  // see one_row
  const T *x;
  __device__ __forceinline__ T gather(int k) const { return __ldg(x + k); }
  __device__ __forceinline__ void add(T &acc, T a, T v) const { acc += a * v; }
};

inline int grid_for(long long work_items, int per_block) {
  long long b = (work_items + per_block - 1) / per_block;
  if (b < 1) b = 1;
  if (b > kMaxBlocks) b = kMaxBlocks;
  return (int)b;
}

}  // namespace pdq

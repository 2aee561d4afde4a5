// Failure-detection self-test: makes bounded device waits run out on purpose,
// without a fault; they must give up after their poll limits, set the fault flag
// and return, leaving the context usable.  loop_sync, the one spin-wait of the
// solver's kernels, runs out in a grid one of whose blocks never reaches it, and
// in the launches of a solve, whose call must report it.  The third is the
// bounded mbarrier wait of a bulk copy; no kernel of the solver waits on one.
#include <cuda_runtime.h>

#include <chrono>
#include <memory>
#include <string>

#include "../../include/pdnqp.h"
#include "common.cuh"
#include "solver.cuh"

namespace pdq {
namespace {

// Block 0 leaves before the barrier: no leader ever releases the others.
__global__ void k_selftest_barrier(unsigned *bar, int *ret) {
  if (blockIdx.x == 0) return;
  unsigned gen = threadIdx.x == 0 ? ld_acquire_gpu(bar + kBarGen) : 0u;
  const bool ok = loop_sync<false>(bar, gen) >= 0;
  if (threadIdx.x == 0) ret[blockIdx.x] = ok ? 1 : 0;
}

// Shared-memory mbarrier: one thread arms it with the byte count that it expects,
// and its phase completes when the bytes have landed.
constexpr unsigned kSpinLimitTx = 1u << 24;  // polls (with a 32 ns sleep)
__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long *bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
// Makes barrier initialisation visible to the copy engine (async proxy).
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned long long *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_test(unsigned long long *bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0u;
}
// Bounded wait of one warp for the phase with the given parity: lane 0 polls
// (and every 64 polls looks at the fault flag), the result is warp-uniform,
// and on success every lane observes the completed phase itself, which makes
// the copied bytes visible to it.  Returns false on a timeout (the fault flag
// is then set) or when another warp has already set the fault flag.
__device__ __forceinline__ bool mbar_wait_warp(unsigned long long *bar, unsigned parity, unsigned *fault) {
  int r = 0;
  if ((threadIdx.x & 31) == 0) {
    for (unsigned it = 0; it <= kSpinLimitTx; ++it) {
      if (mbar_test(bar, parity)) {
        r = 1;
        break;
      }
      if ((it & 63u) == 63u && ld_acquire_gpu(fault) != 0u) break;
      __nanosleep(32);
    }
    if (!r) atomicExch(fault, 1u);
  }
  r = __shfl_sync(0xffffffffu, r, 0);
  if (r)
    for (unsigned it = 0; it <= kSpinLimitTx && !mbar_test(bar, parity); ++it) {
    }
  __syncwarp();
  return r != 0;
}

// One arrival with an expected transaction of 16 bytes and no copy issued:
// the phase never completes.  No asynchronous operation is in flight.
__global__ void k_selftest_tx(unsigned *fault, int *ret) {
  __shared__ unsigned long long bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_init_fence();
  }
  __syncthreads();
  if (threadIdx.x == 0) mbar_arrive_expect_tx(&bar, 16u);
  __syncthreads();
  const bool ok = mbar_wait_warp(&bar, 0u, fault);
  if ((threadIdx.x & 31) == 0) ret[threadIdx.x >> 5] = ok ? 1 : 0;
}

// A solve in the grid form (n = 20,000, an identity Q) whose barrier starts from an
// arrival count that it can never complete: the first launch gives up, the solve
// reports PDNQP_ERR_CUDA, and the next one on the same solver runs to its end.
int selftest_solver(int *gave_up) {
  HostProblem H;
  H.n = 20000;
  H.q_rp.resize(H.n + 1);
  for (int i = 0; i <= H.n; ++i) H.q_rp[i] = i;
  H.q_ci.assign(H.q_rp.begin(), H.q_rp.end() - 1);
  H.q_diag = H.q_ci;
  H.q_v.assign(H.n, 1.0);
  H.a_rp.assign(1, 0);
  H.at_rp.assign(H.n + 1, 0);
  H.c.assign(H.n, -0.5);
  H.lx.assign(H.n, 0.0);
  H.ux.assign(H.n, 1.0);
  std::unique_ptr<SolverBase> s(make_solver_f64(nullptr));
  Params prm;
  std::string err;
  int rc = s->setup(H, prm, &err);
  if (rc < 0) return rc;
  rc = s->jam_barrier();
  if (rc < 0) return rc;
  const int first = s->solve(1e-6, 1e-6, prm, &err), again = s->solve(1e-6, 1e-6, prm, &err);
  *gave_up = first == PDNQP_ERR_CUDA && again == PDNQP_SOLVED ? 1 : 0;
  return 0;
}

}  // namespace
}  // namespace pdq

extern "C" int pdnqp_selftest_wait(int kind, int *gave_up, double *seconds) {
  using namespace pdq;
  if (kind < 0 || kind > 2 || !gave_up) return PDNQP_ERR_ARG;
  if (kind == 2) {
    const auto t0 = std::chrono::steady_clock::now();
    int rc;
    try {
      rc = selftest_solver(gave_up);
    } catch (...) {  // host memory
      rc = PDNQP_ERR_OOM;
    }
    if (seconds) *seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    return rc;
  }
  constexpr int kBlocks = 4, kRet = 8;
  unsigned *bar = nullptr;
  int *ret = nullptr;
  if (cudaMalloc(&bar, kBarWords * sizeof(unsigned)) != cudaSuccess) return PDNQP_ERR_OOM;
  if (cudaMalloc(&ret, kRet * sizeof(int)) != cudaSuccess) {
    cudaFree(bar);
    return PDNQP_ERR_OOM;
  }
  int rc = 0;
  int hret[kRet];
  unsigned hbar[kBarWords];
  const auto t0 = std::chrono::steady_clock::now();
  if (cudaMemset(bar, 0, kBarWords * sizeof(unsigned)) != cudaSuccess ||
      cudaMemset(ret, 0xff, kRet * sizeof(int)) != cudaSuccess) {
    rc = PDNQP_ERR_CUDA;
  } else {
    if (kind == 0)
      k_selftest_barrier<<<kBlocks, kBlock>>>(bar, ret);
    else
      k_selftest_tx<<<1, kBlock>>>(bar + kBarFault, ret);
    if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess ||
        cudaMemcpy(hret, ret, sizeof(hret), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(hbar, bar, sizeof(hbar), cudaMemcpyDeviceToHost) != cudaSuccess)
      rc = PDNQP_ERR_CUDA;
  }
  const double dt = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  if (seconds) *seconds = dt;
  if (rc == 0) {
    // Every waiter reported failure and the fault flag is set.
    bool all = hbar[kBarFault] == 1u;
    const int first = kind == 0 ? 1 : 0, last = kind == 0 ? kBlocks : kBlock / 32;
    for (int b = first; b < last; ++b) all = all && hret[b] == 0;
    *gave_up = all ? 1 : 0;
  }
  cudaFree(bar);
  cudaFree(ret);
  return rc;
}

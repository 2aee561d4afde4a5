// External KKT test of a point (Sec. 4.1) on problem data held in device
// memory: the residuals of Eqs. outer-residuals / outer-scales on the
// original (unscaled) problem, with variable-bound violations counted in r_p.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>

#include "../../include/pdnqp.h"
#include "kkt_kernels.cuh"

namespace pdq {
namespace {

static thread_local std::string g_kkt_err;

int check_problem(const pdnqp_device_problem *P, const double *x, const double *y, const double *out) {
  if (!P || !x || !out) {
    g_kkt_err = "NULL argument";
    return PDNQP_ERR_ARG;
  }
  const int n = P->Q.n_rows, m = P->A.n_rows;
  if (n <= 0 || P->Q.n_cols != n || !P->Q.row_ptr || (P->Q.nnz > 0 && (!P->Q.col_idx || !P->Q.val))) {
    g_kkt_err = "Q must be a square n x n device CSR with n >= 1";
    return PDNQP_ERR_ARG;
  }
  if (P->Q.nnz < 0 || P->Q.nnz > 2147483647LL || P->A.nnz < 0 || P->A.nnz > 2147483647LL) {
    g_kkt_err = "nnz must fit the int32 CSR indices";
    return PDNQP_ERR_ARG;
  }
  if (m < 0 || (m > 0 && (P->A.n_cols != n || !P->A.row_ptr || !P->At.row_ptr || P->At.n_rows != n ||
                          P->At.n_cols != m || !P->l_c || !P->u_c || !y))) {
    g_kkt_err = "A (m x n), At (n x m), l_c, u_c and y are required when m > 0";
    return PDNQP_ERR_ARG;
  }
  if (!P->c || !P->l_x || !P->u_x) {
    g_kkt_err = "c, l_x and u_x are required";
    return PDNQP_ERR_ARG;
  }
  return 0;
}

int launch_kkt(const pdnqp_device_problem *P, const double *x, const double *y, double *out, cudaStream_t s) {
  const int n = P->Q.n_rows, m = P->A.n_rows;
  const KktCsr Q{P->Q.row_ptr, P->Q.col_idx, P->Q.val};
  KktCsr A{nullptr, nullptr, nullptr}, At = A;
  if (m > 0) {
    A = KktCsr{P->A.row_ptr, P->A.col_idx, P->A.val};
    At = KktCsr{P->At.row_ptr, P->At.col_idx, P->At.val};
  }
  // Rows of Q (the matrix that carries the entries) of more than 24 on average:
  // tiles of 8 rows, else of 32 (whose long rows go one at a time).
  const bool lng = P->Q.nnz > 24 * (int64_t)n;
  const int tr = lng ? 8 : 32;
  const long long tiles = ((long long)n + tr - 1) / tr + ((long long)m + tr - 1) / tr;
  // As many blocks as are resident together (3 on each of 152 SMs): a grid of
  // 1216 ran 2.67 waves of unequal length (114 us instead of 105 at n = 1e6).
  const int nb = std::min(grid_for(tiles, kBlock / 32), 3 * 152);
  k_kkt_init<<<1, 32, 0, s>>>(out);
  if (lng)
    k_kkt<true><<<nb, kBlock, 0, s>>>(n, m, Q, At, A, P->c, P->l_c, P->u_c, P->l_x, P->u_x, x, y, out);
  else
    k_kkt<false><<<nb, kBlock, 0, s>>>(n, m, Q, At, A, P->c, P->l_c, P->u_c, P->l_x, P->u_x, x, y, out);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    g_kkt_err = std::string("kernel launch: ") + cudaGetErrorString(e);
    return PDNQP_ERR_CUDA;
  }
  return 0;
}

}  // namespace
}  // namespace pdq

extern "C" {

int pdnqp_kkt_residuals_noalloc(const pdnqp_device_problem *P, const double *x, const double *y, double *out,
                                void *stream) {
  using namespace pdq;
  int rc = check_problem(P, x, y, out);
  if (rc) return rc;
  return launch_kkt(P, x, y, out, (cudaStream_t)stream);
}

int pdnqp_kkt_residuals(const pdnqp_device_problem *P, const double *x, const double *y, double *out,
                        void *stream) {
  using namespace pdq;
  int rc = check_problem(P, x, y, out);
  if (rc) return rc;
  rc = launch_kkt(P, x, y, out, (cudaStream_t)stream);
  const cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
  if (rc) return rc;
  if (e != cudaSuccess) {
    g_kkt_err = std::string("cudaStreamSynchronize: ") + cudaGetErrorString(e);
    return PDNQP_ERR_CUDA;
  }
  return 0;
}

const char *pdnqp_kkt_last_error(void) { return pdq::g_kkt_err.c_str(); }

}  // extern "C"

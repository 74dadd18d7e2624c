// Low-rank preconditioner of Section 3.1 / Algorithm 3 (its SVD, step 4, is in tk_svd.cu).
//
//  * sd_i = sum_j 1/(1 + lambda_i/sigma_j^2) (Section 3.1.2) and the ranks
//    s_i = min(s, ceil(alpha ceil(sd_i))) (step 5), in float64 with the sum
//    taken in ascending j and no contraction, so equal sigma give equal ranks
//    on any IEEE machine.
//  * S_i = diag(1 - sqrt(1/(1 + sigma_j^2/lambda_i))) (step 7) and the apply
//    R_i^-1 x = lambda_i^{-1/2} (x - V_i S_i V_i^T x) (eq. for R^-1, step 8).
#include <algorithm>

#include "tk_lsqr.cuh"

namespace tk {
namespace {

// sd_i and s_i for each lambda (one thread per lambda; sum in ascending j).
__global__ void k_ranks(const double* __restrict__ sigma, int64_t s, const double* __restrict__ lam, int N,
                        double alpha, double* __restrict__ sd_out, int64_t* __restrict__ rank_out) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const double l = lam[i];
  double acc = 0.0;
  for (int64_t j = 0; j < s; ++j) {
    double sg = sigma[j];
    if (sg > 0.0) acc = __dadd_rn(acc, __ddiv_rn(1.0, __dadd_rn(1.0, __ddiv_rn(l, __dmul_rn(sg, sg)))));
  }
  double t = ceil(__dmul_rn(alpha, ceil(acc)));
  int64_t r = (t > (double)s) ? s : (t < 1.0 ? 1 : (int64_t)t);
  if (sd_out) sd_out[i] = acc;
  rank_out[i] = r;
}

// S[l][j] = 1 - sqrt(1/(1 + sigma_j^2/lambda_l)) for j < rank_l, else 0.
template <typename T>
__global__ void k_lr_diag(const double* __restrict__ sigma, int64_t s, const double* __restrict__ lam,
                          const int64_t* __restrict__ rank, T* __restrict__ S) {
  const int l = blockIdx.y;
  const double lv = lam[l];
  const int64_t r = rank[l];
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < s; j += (int64_t)gridDim.x * blockDim.x) {
    double v = 0.0;
    if (j < r) v = 1.0 - sqrt(1.0 / (1.0 + sigma[j] * sigma[j] / lv));
    S[(int64_t)l * s + j] = (T)v;
  }
}

// tmp[k][j] *= S[l_k][j] / sqrt(lambda_l);  invs[k] = 1/sqrt(lambda_l)
template <typename T>
__global__ void k_lr_scale(T* __restrict__ tmp, int64_t s, const T* __restrict__ S, const int* __restrict__ lam_idx,
                           const double* __restrict__ lam, double* __restrict__ invs) {
  const int k = blockIdx.y;
  const int l = lam_idx[k];
  const double is = 1.0 / sqrt(lam[l]);
  if (blockIdx.x == 0 && threadIdx.x == 0) invs[k] = is;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < s; j += (int64_t)gridDim.x * blockDim.x)
    tmp[(int64_t)k * s + j] = (T)((double)tmp[(int64_t)k * s + j] * (double)S[(int64_t)l * s + j] * is);
}

}  // namespace

tk_status lowrank_ranks_dev(const double* sigma, int64_t s, const double* lam_dev, int N, double alpha,
                            double* sd_dev, int64_t* rank_dev, cudaStream_t st) {
  if (N <= 0) return TK_OK;
  k_ranks<<<cdiv(N, 128), 128, 0, st>>>(sigma, s, lam_dev, N, alpha, sd_dev, rank_dev);
  TK_LAUNCH_CHECK();
  return TK_OK;
}

template <typename T>
tk_status lowrank_diag_dev(const double* sigma, int64_t s, const double* lam_dev, const int64_t* rank_dev, int N,
                           T* S, cudaStream_t st) {
  if (N <= 0 || s <= 0) return TK_OK;
  dim3 g((unsigned)std::min<int64_t>(cdiv(s, 256), 64), (unsigned)N);
  k_lr_diag<T><<<g, 256, 0, st>>>(sigma, s, lam_dev, rank_dev, S);
  TK_LAUNCH_CHECK();
  return TK_OK;
}
template tk_status lowrank_diag_dev<double>(const double*, int64_t, const double*, const int64_t*, int, double*,
                                            cudaStream_t);
template tk_status lowrank_diag_dev<float>(const double*, int64_t, const double*, const int64_t*, int, float*,
                                           cudaStream_t);

template <typename T>
tk_status lr_apply(int count, int64_t n, int64_t s, const T* V, const T* S, const int* lam_idx,
                   const double* lam_dev, const T* in, T* out, T* tmp, double* invs, cudaStream_t st) {
  if (count <= 0) return TK_OK;
  // tmp = in V  (count x s)
  TK_TRY((gemm<T, T, T>(false, false, count, s, n, in, n, V, s, tmp, s, 1.0, nullptr, nullptr, 0, st)));
  dim3 g((unsigned)std::max<int64_t>(1, std::min<int64_t>(cdiv(s, 256), 64)), (unsigned)count);
  k_lr_scale<T><<<g, 256, 0, st>>>(tmp, s, S, lam_idx, lam_dev, invs);
  TK_LAUNCH_CHECK();
  // out = -tmp V^T + invs * in
  TK_TRY((gemm<T, T, T>(false, true, count, n, s, tmp, s, V, s, out, n, -1.0, invs, in, n, st)));
  return TK_OK;
}
template tk_status lr_apply<double>(int, int64_t, int64_t, const double*, const double*, const int*, const double*,
                                    const double*, double*, double*, double*, cudaStream_t);
template tk_status lr_apply<float>(int, int64_t, int64_t, const float*, const float*, const int*, const double*,
                                   const float*, float*, float*, double*, cudaStream_t);

}  // namespace tk

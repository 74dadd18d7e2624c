// Low-rank preconditioner of Section 3.1 / Algorithm 3 (its SVD, step 4, is in tk_svd.cu).
//
//  * sd_i = sum_j 1/(1 + lambda_i/sigma_j^2) (Section 3.1.2) and the ranks
//    s_i = min(s, ceil(alpha ceil(sd_i))) (step 5), in float64 with the sum
//    taken in ascending j and no contraction, so equal sigma give equal ranks
//    on any IEEE machine.
//  * S_i = diag(1 - sqrt(1/(1 + sigma_j^2/lambda_i))) (step 7) and the apply
//    R_i^-1 x = lambda_i^{-1/2} (x - V_i S_i V_i^T x) (eq. for R^-1, step 8).
#include <algorithm>

#include "tk_gemm_tiles.cuh"
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

// The apply out_k = l^{-1/2} (in_k - V S_l V^T in_k) in three launches.  V (n x s) is a few MB: it is
// read from L2 once per LR_NL slots and product, and the grids fill the GPU (as general products of
// 16 x 1000 x 462 float64 the two ran on 15 and 32 CTAs: 420 us an apply, now 45).
constexpr int LR_ROWS = 64;  // rows of `in` staged at a time

// part[z][k][c] = sum over the rows i of split z of in[k][i] V[i][c]: CTA = 32 columns x 8 row groups,
// NL slots (blockIdx.z), one accumulator per slot and thread.
template <typename T, int NL>
__global__ void __launch_bounds__(256)
    k_lr_tv(const T* __restrict__ in, int count, int64_t n, const T* __restrict__ V, int64_t s, int64_t rows_per,
            double* __restrict__ part) {
  __shared__ __align__(16) T xs[LR_ROWS][NL];
  __shared__ T red[8][NL][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t c = (int64_t)blockIdx.x * 32 + tx;
  const int k0 = blockIdx.z * NL;
  const int64_t rb = (int64_t)blockIdx.y * rows_per, re = rb + rows_per < n ? rb + rows_per : n;
  T acc[NL];
#pragma unroll
  for (int l = 0; l < NL; ++l) acc[l] = T(0);
  for (int64_t i0 = rb; i0 < re; i0 += LR_ROWS) {
    __syncthreads();
    for (int idx = threadIdx.x; idx < LR_ROWS * NL; idx += 256) {
      const int l = idx / LR_ROWS, r = idx % LR_ROWS;
      xs[r][l] = (k0 + l < count && i0 + r < re) ? in[(int64_t)(k0 + l) * n + i0 + r] : T(0);
    }
    __syncthreads();
    const int nr = (int)(re - i0 < LR_ROWS ? re - i0 : LR_ROWS);
    T v[LR_ROWS / 8];
#pragma unroll
    for (int q = 0; q < LR_ROWS / 8; ++q) {
      const int r = ty + 8 * q;
      v[q] = (c < s && r < nr) ? V[(i0 + r) * s + c] : T(0);
    }
#pragma unroll
    for (int q = 0; q < LR_ROWS / 8; ++q)
#pragma unroll
      for (int l = 0; l < NL; ++l) acc[l] = fma(v[q], xs[ty + 8 * q][l], acc[l]);
  }
#pragma unroll
  for (int l = 0; l < NL; ++l) red[ty][l][tx] = acc[l];
  __syncthreads();
  for (int l = ty; l < NL; l += 8) {
    if (k0 + l >= count || c >= s) continue;
    T t = red[0][l][tx];
#pragma unroll
    for (int q = 1; q < 8; ++q) t += red[q][l][tx];
    part[((int64_t)blockIdx.y * count + k0 + l) * s + c] = (double)t;
  }
}

// t[k][c] = S[l_k][c] / sqrt(lambda_l) sum_z part[z][k][c];  invs[k] = 1 / sqrt(lambda_l)
template <typename T>
__global__ void __launch_bounds__(256)
    k_lr_scale(const double* __restrict__ part, int splits, int count, int64_t s, const T* __restrict__ S,
               const int* __restrict__ lam_idx, const double* __restrict__ lam, T* __restrict__ t,
               double* __restrict__ invs) {
  const int k = blockIdx.y;
  const int l = lam_idx[k];
  const double is = 1.0 / sqrt(lam[l]);
  if (blockIdx.x == 0 && threadIdx.x == 0) invs[k] = is;
  const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= s) return;
  double acc = 0.0;
#pragma unroll 4
  for (int z = 0; z < splits; ++z) acc += part[((int64_t)z * count + k) * s + j];
  t[(int64_t)k * s + j] = (T)(acc * (double)S[(int64_t)l * s + j] * is);
}

// out[k][i] = invs[k] in[k][i] - sum_c t[k][c] V[i][c]: a warp takes two rows, NL slots' t in shared
// memory; the 2 NL sums are folded over the warp together.
template <typename T, int NL>
__global__ void __launch_bounds__(256)
    k_lr_vt(const T* __restrict__ in, int count, int64_t n, const T* __restrict__ V, int64_t s,
            const T* __restrict__ t, const double* __restrict__ invs, T* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char lr_sm[];
  T* ts = reinterpret_cast<T*>(lr_sm);  // [NL][s]
  const int k0 = blockIdx.y * NL;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t idx = threadIdx.x; idx < NL * s; idx += 256)
    ts[idx] = k0 + idx / s < count ? t[(int64_t)k0 * s + idx] : T(0);
  __syncthreads();
  for (int64_t i = ((int64_t)blockIdx.x * 8 + w) * 2; i < n; i += (int64_t)gridDim.x * 16) {
    const T* r0 = V + i * s;
    const T* r1 = V + (i + 1 < n ? i + 1 : i) * s;
    T acc[2 * NL];
#pragma unroll
    for (int q = 0; q < 2 * NL; ++q) acc[q] = T(0);
#pragma unroll 4
    for (int64_t c = lane; c < s; c += 32) {
      const T a = r0[c], b = r1[c];
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        const T tv = ts[l * s + c];
        acc[l] = fma(a, tv, acc[l]);
        acc[NL + l] = fma(b, tv, acc[NL + l]);
      }
    }
    int which;
    const T sum = tiles::warp_sum_rows<T, 2 * NL>(acc, &which);
    const int l = which % NL;
    const int64_t r = i + which / NL;
    if ((lane & (32 / (2 * NL) - 1)) == 0 && k0 + l < count && r < n)
      out[(int64_t)(k0 + l) * n + r] = (T)(invs[k0 + l] * (double)in[(int64_t)(k0 + l) * n + r] - (double)sum);
  }
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

template <typename T, int NL>
static tk_status lr_apply_nl(int count, int64_t n, int64_t s, const T* V, const T* S, const int* lam_idx,
                             const double* lam_dev, const T* in, T* out, T* tmp, double* invs, double* part,
                             int64_t part_len, cudaStream_t st) {
  const int64_t groups = cdiv(count, NL), ct = cdiv(s, 32);
  // two CTAs per SM, at least LR_ROWS rows to a split, the planes within `part`
  const int64_t want = cdiv(2 * 152, ct * groups);
  const int64_t splits = std::max<int64_t>(1, std::min<int64_t>({want, cdiv(n, LR_ROWS), part_len / (count * s)}));
  const int64_t per = cdiv(cdiv(n, splits), LR_ROWS) * LR_ROWS;
  const int sp = (int)cdiv(n, per);
  k_lr_tv<T, NL><<<dim3((unsigned)ct, (unsigned)sp, (unsigned)groups), 256, 0, st>>>(in, count, n, V, s, per, part);
  TK_LAUNCH_CHECK();
  k_lr_scale<T><<<dim3((unsigned)cdiv(s, 256), (unsigned)count), 256, 0, st>>>(part, sp, count, s, S, lam_idx, lam_dev,
                                                                              tmp, invs);
  TK_LAUNCH_CHECK();
  constexpr int kCap = 160 * 1024;  // one cap: host threads launch concurrently
  auto kern = k_lr_vt<T, NL>;
  TK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kCap));
  const unsigned gx = (unsigned)std::max<int64_t>(1, std::min<int64_t>(cdiv(n, 16), cdiv(4 * 152, groups)));
  kern<<<dim3(gx, (unsigned)groups), 256, sizeof(T) * NL * (size_t)s, st>>>(in, count, n, V, s, tmp, invs, out);
  TK_LAUNCH_CHECK();
  return TK_OK;
}

template <typename T>
tk_status lr_apply(int count, int64_t n, int64_t s, const T* V, const T* S, const int* lam_idx,
                   const double* lam_dev, const T* in, T* out, T* tmp, double* invs, double* part, int64_t part_len,
                   cudaStream_t st) {
  if (count <= 0) return TK_OK;
  // 8 slots share a read of V while their t fits in shared memory (s <= 2560 in float64), else 2
  if (sizeof(T) * 8 * (size_t)s <= 160 * 1024)
    return lr_apply_nl<T, 8>(count, n, s, V, S, lam_idx, lam_dev, in, out, tmp, invs, part, part_len, st);
  return lr_apply_nl<T, 2>(count, n, s, V, S, lam_idx, lam_dev, in, out, tmp, invs, part, part_len, st);
}
template tk_status lr_apply<double>(int, int64_t, int64_t, const double*, const double*, const int*, const double*,
                                    const double*, double*, double*, double*, double*, int64_t, cudaStream_t);
template tk_status lr_apply<float>(int, int64_t, int64_t, const float*, const float*, const int*, const double*,
                                   const float*, float*, float*, double*, double*, int64_t, cudaStream_t);

}  // namespace tk

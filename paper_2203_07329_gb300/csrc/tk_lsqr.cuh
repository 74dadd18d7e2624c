// Batched preconditioned LSQR engine (internal).
#pragma once

#include <type_traits>
#include <vector>

#include "tk_internal.cuh"

namespace tk {

// Per-slot LSQR scalars (device resident).
struct Scal {
  double alpha, beta, rhobar, phibar, anorm2, bnorm, lam, sqrtl, coef, rnorm, arnorm, ynorm;
  int iters, istop, lam_idx, pad;
};

struct LsqrResult {
  int lam_idx, iters, istop;
  double rnorm, arnorm;
};

// Low-rank preconditioner apply (Section 3.1, eq. for R^-1):
// out_k = l^{-1/2} (in_k - V diag(S_l) V^T in_k) for each listed row k, with
// l = lam_idx[k]; V is n x s (row-major), S is N_lam x s (zero past s_l); part: part_len >= count s doubles of
// scratch (the split sums of V^T in).
template <typename T>
tk_status lr_apply(int count, int64_t n, int64_t s, const T* V, const T* S, const int* lam_idx,
                   const double* lam_dev, const T* in, T* out, T* tmp, double* invs, double* part, int64_t part_len,
                   cudaStream_t st);

// sd_i, s_i of Algorithm 3 step 5 (device in/out) and the S_i rows (step 7).
tk_status lowrank_ranks_dev(const double* sigma, int64_t s, const double* lam_dev, int N, double alpha,
                            double* sd_dev, int64_t* rank_dev, cudaStream_t st);
template <typename T>
tk_status lowrank_diag_dev(const double* sigma, int64_t s, const double* lam_dev, const int64_t* rank_dev, int N,
                           T* S, cudaStream_t st);

// One slot's Golub-Kahan v-step (Paige & Saunders' LSQR): Vraw holds M^T u
// (length nv).  v' = Vraw - beta v, alpha = ||v'||, then the Givens rotation,
// the y and w updates and the stopping tests (istop 1: the residual test, 2:
// the normal-equation test, 5: non-finite, 7: iteration cap).  init: the first
// v (alpha_1 v_1 = M^T u_1), w = v, y = 0.
struct VGivens {
  double ainv, t1, t2;  // 1 / alpha, phi / rho, theta / rho
  double c, rhobar, phibar;
};
// Roots and quotients through reciprocal roots: a float64 division or root is a dependent chain of a
// dozen instructions on a slow pipe, and this is on the critical path of every step.
__device__ __forceinline__ VGivens vstep_givens(const Scal& q, double alpha, double ainv) {
  VGivens g;
  const double r2 = fma(q.rhobar, q.rhobar, q.beta * q.beta);
  const double rinv = r2 > 0.0 ? rsqrt(r2) : 0.0;
  g.c = r2 > 0.0 ? q.rhobar * rinv : 1.0;
  const double sn = q.beta * rinv;
  g.rhobar = -g.c * alpha;
  g.phibar = sn * q.phibar;
  g.t1 = g.c * q.phibar * rinv;
  g.t2 = sn * alpha * rinv;
  g.ainv = ainv;
  return g;
}
__device__ __forceinline__ void vstep_init_scal(Scal& q, double alpha) {
  q.alpha = alpha;
  q.rhobar = alpha;
  q.coef = (q.beta > 0.0) ? -alpha / q.beta : 0.0;
  q.arnorm = alpha * q.beta;
  if (alpha == 0.0 && q.istop == 0) q.istop = 1;  // b orthogonal to range(M): y = 0 is exact
  if (!isfinite(alpha)) q.istop = 5;
}
__device__ __forceinline__ void vstep_finish_scal(Scal& q, const VGivens& g, double alpha, double ynorm, double atol,
                                                  double btol, int maxiter) {
  const double beta = q.beta;
  q.alpha = alpha;
  q.rhobar = g.rhobar;
  q.phibar = g.phibar;
  q.iters += 1;
  q.coef = beta > 0.0 ? -alpha / beta : 0.0;
  const double rnorm = g.phibar;
  const double arnorm = g.phibar * alpha * fabs(g.c);
  const double anorm = sqrt(q.anorm2);
  q.rnorm = rnorm;
  q.arnorm = arnorm;
  q.ynorm = ynorm;
  int istop = 0;
  if (!isfinite(alpha) || !isfinite(beta) || !isfinite(ynorm)) istop = 5;
  else if (rnorm == 0.0) istop = 1;
  else if (arnorm <= atol * (anorm * rnorm)) istop = 2;
  else if (rnorm <= btol * q.bnorm + atol * anorm * ynorm) istop = 1;
  else if (q.iters >= maxiter) istop = 7;
  q.istop = istop;
}

// The step by CL CTAs of a cluster (CL = 1: a plain block), this CTA taking every CL-th block of
// values; sh: 32 doubles, red: 2 doubles of shared memory that the peers read.
template <typename T, int CL>
__device__ __forceinline__ void vstep_block(const T* __restrict__ Vraw, T* __restrict__ V, T* __restrict__ W,
                                            T* __restrict__ Y, int64_t nv, Scal* __restrict__ sq,
                                            double* __restrict__ coef_out, double atol, double btol, int maxiter,
                                            int init, double* sh, double* red) {
  Scal q = *sq;
  if (!init && q.istop != 0) return;  // retired inside a chunk of steps: left as it is (every CTA returns)
  const double beta = q.beta;
  int rank = 0;
  if constexpr (CL > 1) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  // sum over the cluster, in rank order; slot: a fresh entry of red for each sum
  auto cluster_sum = [&](double v, int slot) -> double {
    v = block_sum(v, sh);
    if constexpr (CL > 1) {
      if (threadIdx.x == 0) red[slot] = v;
      asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
      v = 0.0;
#pragma unroll
      for (int r = 0; r < CL; ++r) v += *static_cast<double*>(__cluster_map_shared_rank(red + slot, r));
    }
    return v;
  };
  const int64_t first = (int64_t)rank * blockDim.x + threadIdx.x, stride = (int64_t)CL * blockDim.x;
  __shared__ double bc[3];  // 1 / alpha, phi / rho, theta / rho from the first warp: every warp computing
                            // them would queue for the float64 pipe (9.5 us a step at n = 256, now 6.3)
  // v' = Vraw - beta v  (init: v' = Vraw)
  double acc = 0.0;
#pragma unroll 4
  for (int64_t j = first; j < nv; j += stride) {
    double v = (double)Vraw[j];
    if (!init) v = fma(-beta, (double)V[j], v);
    V[j] = (T)v;
    acc = fma(v, v, acc);
  }
  const double a2 = cluster_sum(acc, 0);
  double alpha = 0.0;
  VGivens g;
  if (threadIdx.x < 32) {
    alpha = sqrt(a2);
    const double ainv = a2 > 0.0 ? rsqrt(a2) : 0.0;
    g = vstep_givens(q, alpha, ainv);
    if (threadIdx.x == 0) {
      bc[0] = g.ainv;
      bc[1] = g.t1;
      bc[2] = g.t2;
    }
  }
  __syncthreads();
  const double ainv = bc[0], t1 = bc[1], t2 = bc[2];
  if (init) {
    for (int64_t j = first; j < nv; j += stride) {
      T v = (T)((double)V[j] * ainv);
      V[j] = v;
      W[j] = v;
      Y[j] = T(0);
    }
    if (rank == 0 && threadIdx.x == 0) {
      vstep_init_scal(q, alpha);
      *sq = q;
      if (coef_out) *coef_out = q.coef;
    }
  } else {
    double yy = 0.0;
#pragma unroll 4
    for (int64_t j = first; j < nv; j += stride) {
      double v = (double)V[j] * ainv;
      double w = (double)W[j];
      double y = fma(t1, w, (double)Y[j]);
      w = fma(-t2, w, v);
      V[j] = (T)v;
      W[j] = (T)w;
      Y[j] = (T)y;
      yy = fma(y, y, yy);
    }
    const double y2 = cluster_sum(yy, 1);
    if (rank == 0 && threadIdx.x == 0) {
      const double ynorm = sqrt(y2);
      vstep_finish_scal(q, g, alpha, ynorm, atol, btol, maxiter);
      *sq = q;
      if (coef_out) *coef_out = q.coef;
    }
  }
  // no CTA leaves while a peer may still read its sums
  if constexpr (CL > 1)
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The replays of one solve: chunks of LSQR steps captured once per slot count, and the stream they run
// on (the caller's may be the legacy default stream, which cannot be captured).
struct StepGraphs {
  cudaStream_t st = nullptr;
  cudaEvent_t ev = nullptr;
  struct Entry {
    int slots;
    cudaGraphExec_t exec;
    size_t kernels;
  };
  std::vector<Entry> entries;
  StepGraphs() = default;
  StepGraphs(const StepGraphs&) = delete;
  StepGraphs& operator=(const StepGraphs&) = delete;
  ~StepGraphs() {
    if (st) cudaStreamSynchronize(st);
    for (auto& e : entries) cudaGraphExecDestroy(e.exec);
    if (ev) cudaEventDestroy(ev);
    if (st) cudaStreamDestroy(st);
  }
};

template <typename T>
struct Lsqr {
  // problem: A (m x n, row stride lda) in the compute type
  const T* A = nullptr;
  int64_t m = 0, n = 0, lda = 0;
  // bytes per element of A in the caller's dtype (the profiler's algorithmic bytes of one A pass)
  double a_es = sizeof(T);
  bool under = false;
  // preconditioner: per-lambda Cholesky factors R + l*rstride, or low rank
  tk_precond prec_kind = TK_PRECOND_CHOL;
  const T* R = nullptr;
  int64_t ldr = 0, rstride = 0;
  // explicit inverse: Mi = R^-1, Mti = R^-T (row stride ldm, matrix stride
  // mstride); when set it replaces the substitutions with R (overdetermined)
  const T* Mi = nullptr;
  const T* Mti = nullptr;
  int64_t ldm = 0, mstride = 0;
  int64_t lr_s = 0;
  const T* lrV = nullptr;
  const T* lrS = nullptr;
  // parameters
  int N_cap = 0;
  double atol = 1e-14, btol = 1e-14;
  int maxiter = 500;
  cudaStream_t st = nullptr;
  // workspace
  int64_t nv = 0;
  int splits = 1;      // split-K capacity of part_g
  int cur_splits = 1;  // splits of the last A^T U product (the tuned count, <= splits)
  T *V = nullptr, *W = nullptr, *Y = nullptr, *Vraw = nullptr, *Ut = nullptr, *Tt = nullptr, *Ub = nullptr,
    *xtmp = nullptr, *lr_tmp = nullptr;
  int* arrivals = nullptr;  // N_cap counters of the norm kernel, zero between launches
  double *part_u = nullptr, *part_g = nullptr, *coef_buf = nullptr, *lr_inv = nullptr, *trsv_p = nullptr;
  Scal* sc = nullptr;
  int* slot_lam = nullptr;
  int* idx_buf = nullptr;
  const double* lam_all = nullptr;
  // tensor-core products (float32 engine only): AT = float32 A^T (n x m)
  bool tc = false;
  const T* AT = nullptr;
  void* tc_scratch = nullptr;
  // products from the digit planes of A on the tensor cores: the first 4 digits (float32 engine) or
  // all 8 (float64 engine)
  bool oz = false;
  OzMat oz_A;
  int* oz_err = nullptr;
  void* oz_q = nullptr;  // slices of the lambda-major vector of a product
  int* oz_e = nullptr;
  // A digit product reads 8 (float32 engine) or 16 bytes (float64) per element of A whatever the
  // number of lambdas; the SIMT products read 4 or 8 bytes but their work grows with it.  Float32: the
  // digits pay off for large A and more than 16 active lambdas.  Float64: the pipe (1.2 TFLOP/s) takes
  // 1.7 ps per element and lambda, the digits 2.7 ps per element, and the pipe's smallest tile does the
  // work of 8 lambdas (a single lambda of 30000 x 1000: 560 us against 105; 4096 x 256, 8 lambda: 37 us
  // against 20): whenever A has 2^19 elements (2000 x 64, one lambda: 15 us on the pipe, 20 from digits).
  bool use_oz(int count) const {
    if (!oz || !oz_A.planes) return false;
    if (std::is_same<T, double>::value) return (int64_t)m * n >= (int64_t(1) << 19);
    return (int64_t)m * n > (int64_t(1) << 24) && count > 16;
  }
  // both products of an overdetermined step in one kernel over one read of
  // the digits (n <= 2048, at most 32 lambda per launch)
  bool oz_fused = false;
  bool use_fused(int count) const { return oz_fused && !under && use_oz(count) && oz_fused_supported(m, n, count); }

  static size_t workspace(int64_t m, int64_t n, int N_cap, bool under, int64_t lr_s);
  void carve(Arena& a);
  // Solve for `count` lambdas (indices lam_ids_dev[k] into lam_dev).  The
  // right-hand side of the k-th listed lambda is [b + k*ldbt; (bbot + k*ldbb) / sqrt(l)]
  // (overdetermined; ldbt = 0 shares b; b or bbot null = zero block) or b
  // (underdetermined).  Writes (or adds) x_l into Xout + l*ldo.
  tk_status run(const double* b, int64_t ldbt, const double* bbot, int64_t ldbb, const int* lam_ids_dev,
                const double* lam_dev, int count, double* Xout, int64_t ldo, bool accumulate,
                std::vector<LsqrResult>& results);
  tk_status apply_prec(bool transposed, const T* in, T* out, int count, int64_t len);
  tk_status prod_aw(const T* Win, int64_t ldw, T* C, const double* beta, int count);
  tk_status prod_atu(const T* Uin, int count);
  tk_status prod_fused(const T* Win, T* C, const double* beta, int count);
  tk_status norm(int nact);
  // one LSQR step for slots 0..nact-1; `count` of them, replayed from a graph
  tk_status step(int nact);
  tk_status replay(int nact, int count);
  StepGraphs graphs;
};

}  // namespace tk

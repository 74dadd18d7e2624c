// Device bodies of the float32 LSQR products for at most 16 lambda, shared by
// the single-problem kernels (tk_lm.cu) and the grouped engine (tk_group.cu).
// Both read the float32 A once in 16-byte vectors along its rows and keep the
// lambda-side operand on chip:
//  * aw_rows: store(l, i, sum_k W[l][k] A[i][k]) for the 4-row
//    groups g_first, g_first + g_stride, ... < g_end, one warp per group at a
//    time; W (zero-padded to NL x n_pad) is in shared memory (load_w); each lane
//    takes 4 consecutive k of every 128, the next 128 loaded while the current
//    ones are used; the 4 NL dot products per lane are added across the warp by
//    halving exchanges (each step keeps half of the values and adds the
//    partner's other half), then written.
//  * atu_cols: out[l][c] = sum over rows rb <= i < re of U[l][i] A[i][c] for the
//    block's columns, CW per thread (NL x CW accumulators, 8 rows' loads in flight);
//    a block with fewer columns than 256 CW splits its rows over groups of threads,
//    whose sums meet in shared memory; the rows' U values are staged in shared memory
//    ([row][lambda], read as broadcasts).  Every thread of the block must call it.
#pragma once
#include "tk_internal.cuh"

namespace tk {
namespace lmb {

constexpr int kRows = 4;          // rows of A per warp (aw)
constexpr int kAtuThreads = 256;  // threads of an atu block
constexpr int kAtuRB = 128;       // rows of U staged at a time (atu)
constexpr int kAwSmemCap = 200 * 1024;  // W's column chunk in shared memory (aw)

// Columns of W (and A) per chunk of the aw product: the most, in 128s, whose NL x chunk floats fit
__host__ __device__ inline int64_t aw_chunk(int nl, int64_t n) {
  const int64_t fit = (int64_t)kAwSmemCap / (4 * nl) / 128 * 128;
  const int64_t n_pad = (n + 127) / 128 * 128;
  return n_pad < fit ? n_pad : fit;
}

__device__ __forceinline__ float dot4(float4 a, float4 b, float acc) {
  acc = fmaf(a.x, b.x, acc);
  acc = fmaf(a.y, b.y, acc);
  acc = fmaf(a.z, b.z, acc);
  return fmaf(a.w, b.w, acc);
}

// 4 consecutive floats of a row from column k (zero past `len`); vector load when allowed
__device__ __forceinline__ float4 load4(const float* __restrict__ row, int64_t k, int64_t len, bool vec) {
  if (vec && k + 3 < len) return __ldg(reinterpret_cast<const float4*>(row + k));
  float e[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) e[t] = k + t < len ? __ldg(row + k + t) : 0.f;
  return make_float4(e[0], e[1], e[2], e[3]);
}

// ws[l][k] = W[l][k] for l < count, k < n, zero elsewhere (NL x n_pad); the caller synchronizes
template <int NL>
__device__ __forceinline__ void load_w(float* ws, const float* __restrict__ W, int64_t ldw, int count, int64_t n,
                                       int64_t n_pad) {
  for (int64_t idx = threadIdx.x; idx < (int64_t)NL * n_pad; idx += blockDim.x) {
    const int l = (int)(idx / n_pad);
    const int64_t k = idx % n_pad;
    ws[idx] = (l < count && k < n) ? W[(int64_t)l * ldw + k] : 0.f;
  }
}

// the store of an LSQR product: C[l][i] = v (+ beta_l C[l][i]), or += v for a later chunk of columns
struct AwStore {
  float* C;
  int64_t ldc;
  const double* beta;
  bool first;
  __device__ __forceinline__ void operator()(int l, int64_t i, float v) const {
    float* c = C + (int64_t)l * ldc + i;
    double val = (double)v;
    if (!first) val += (double)*c;
    else if (beta) val += beta[l] * (double)*c;
    *c = (float)val;
  }
};

template <int NL, typename Store>
__device__ __forceinline__ void aw_rows(const float* ws, int64_t n_pad, const float* __restrict__ A, int64_t lda,
                                        int64_t m, int64_t n, int count, const Store& store, bool vec,
                                        int64_t g_first, int64_t g_stride, int64_t g_end) {
  constexpr int LM_ROWS = kRows;
  const int lane = threadIdx.x & 31;
  const int nj = (int)(n_pad / 128);
  for (int64_t g = g_first; g < g_end; g += g_stride) {
    const int64_t i0 = g * LM_ROWS;
    const float* rows[LM_ROWS];
#pragma unroll
    for (int r = 0; r < LM_ROWS; ++r) rows[r] = A + (i0 + r < m ? i0 + r : i0) * lda;
    const int rmax = (int)(m - i0 < LM_ROWS ? m - i0 : LM_ROWS);
    float acc[LM_ROWS][NL];
#pragma unroll
    for (int r = 0; r < LM_ROWS; ++r)
#pragma unroll
      for (int l = 0; l < NL; ++l) acc[r][l] = 0.f;
    float4 cur[LM_ROWS], nxt[LM_ROWS];
#pragma unroll
    for (int r = 0; r < LM_ROWS; ++r)
      cur[r] = r < rmax ? load4(rows[r], 4 * lane, n, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
    for (int j = 0; j < nj; ++j) {
      const int64_t k = (int64_t)128 * j + 4 * lane;
      if (j + 1 < nj) {
#pragma unroll
        for (int r = 0; r < LM_ROWS; ++r)
          nxt[r] = r < rmax ? load4(rows[r], k + 128, n, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        const float4 w4 = *reinterpret_cast<const float4*>(ws + (int64_t)l * n_pad + k);
#pragma unroll
        for (int r = 0; r < LM_ROWS; ++r) acc[r][l] = dot4(cur[r], w4, acc[r][l]);
      }
#pragma unroll
      for (int r = 0; r < LM_ROWS; ++r) cur[r] = nxt[r];
    }
    // add the V = 4 NL values across the warp: each halving step keeps half (the lanes with bit s
    // set keep the upper half) and adds the partner's copy of it; once one value is left, plain steps
    constexpr int V = LM_ROWS * NL;
    float v[V];
#pragma unroll
    for (int r = 0; r < LM_ROWS; ++r)
#pragma unroll
      for (int l = 0; l < NL; ++l) v[r * NL + l] = acc[r][l];
    int nv = V, qbase = 0;
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) {
      if (nv > 1) {
        const int half = nv / 2;
        const bool up = (lane & s) != 0;
#pragma unroll
        for (int q = 0; q < V / 2; ++q) {
          if (q < half) {
            const float send = up ? v[q] : v[q + half];
            const float keep = up ? v[q + half] : v[q];
            v[q] = keep + __shfl_xor_sync(0xffffffffu, send, s);
          }
        }
        if (up) qbase += half;
        nv = half;
      } else {
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], s);
      }
    }
    // lane holds values qbase .. qbase + nv - 1 (V >= 32: 2 or 1 per lane; V = 16: the same value on
    // two lanes, written by the one with bit 0 clear)
    const bool writer = V >= 32 || (lane & 1) == 0;
    if (writer) {
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        if (t < nv) {
          const int q = qbase + t, r = q / NL, l = q % NL;
          const int64_t i = i0 + r;
          if (i < m && l < count) store(l, i, v[t]);
        }
      }
    }
  }
}

// CW consecutive floats of a row from column k (zero past `len`); vector load when allowed
template <int CW>
__device__ __forceinline__ void loadv(const float* __restrict__ row, int64_t k, int64_t len, bool vec, float (&o)[CW]) {
  if (vec && k + CW - 1 < len) {
    if constexpr (CW == 4) {
      const float4 f = __ldg(reinterpret_cast<const float4*>(row + k));
      o[0] = f.x; o[1] = f.y; o[2] = f.z; o[3] = f.w;
    } else {
      const float2 f = __ldg(reinterpret_cast<const float2*>(row + k));
      o[0] = f.x; o[1] = f.y;
    }
    return;
  }
#pragma unroll
  for (int t = 0; t < CW; ++t) o[t] = k + t < len ? __ldg(row + k + t) : 0.f;
}

// Shared memory of an atu block: the staged U values and the row groups' sums (4 lambda at a time).
template <int NL, int CW>
struct AtuSmem {
  float us[kAtuRB][NL];
  float red[4 * CW][kAtuThreads];
};

// The block's columns c0 .. c0 + CW kAtuThreads - 1 (those < n), rows rb .. re - 1.  CW columns per
// thread (4 for <= 8 lambda, 2 for 16: NL x CW accumulators), 8 rows' loads in flight.
template <int NL, int CW>
__device__ __forceinline__ void atu_cols(AtuSmem<NL, CW>& S, const float* __restrict__ A, int64_t lda, int64_t n,
                                         const float* __restrict__ U, int64_t ldu, int count, int64_t rb, int64_t re,
                                         int64_t c0, double* __restrict__ out, bool vec) {
  constexpr int RU = 8;
  // cg threads across the columns (whole warps), rg groups of rows
  const int64_t cols = n - c0 < (int64_t)CW * kAtuThreads ? n - c0 : (int64_t)CW * kAtuThreads;
  const int cg = (int)((cols + 32 * CW - 1) / (32 * CW)) * 32, rg = kAtuThreads / cg;
  const int g = threadIdx.x / cg;
  const int64_t c = g < rg ? c0 + (int64_t)CW * (threadIdx.x % cg) : n;
  float acc[NL][CW];
#pragma unroll
  for (int l = 0; l < NL; ++l)
#pragma unroll
    for (int t = 0; t < CW; ++t) acc[l][t] = 0.f;
  for (int64_t i0 = rb; i0 < re; i0 += kAtuRB) {
    const int nr = (int)(re - i0 < kAtuRB ? re - i0 : kAtuRB);
    __syncthreads();  // the previous rows' U values are no longer read
    for (int idx = threadIdx.x; idx < kAtuRB * NL; idx += kAtuThreads) {
      const int l = idx / kAtuRB, r = idx % kAtuRB;
      S.us[r][l] = (l < count && r < nr) ? U[(int64_t)l * ldu + i0 + r] : 0.f;
    }
    __syncthreads();
    if (c < n) {
      for (int r = g * RU; r < nr; r += rg * RU) {
        float a[RU][CW];
#pragma unroll
        for (int q = 0; q < RU; ++q) {
          if (r + q < nr) loadv<CW>(A + (i0 + r + q) * lda, c, n, vec, a[q]);
          else {
#pragma unroll
            for (int t = 0; t < CW; ++t) a[q][t] = 0.f;  // us is zero there too
          }
        }
#pragma unroll
        for (int q = 0; q < RU; ++q) {
#pragma unroll
          for (int l4 = 0; l4 < NL / 4; ++l4) {
            const float4 u4 = *reinterpret_cast<const float4*>(&S.us[r + q][4 * l4]);
            const float uu[4] = {u4.x, u4.y, u4.z, u4.w};
#pragma unroll
            for (int t4 = 0; t4 < 4; ++t4)
#pragma unroll
              for (int t = 0; t < CW; ++t) acc[4 * l4 + t4][t] = fmaf(uu[t4], a[q][t], acc[4 * l4 + t4][t]);
          }
        }
      }
    }
  }
  if (rg == 1) {
    if (c < n) {
#pragma unroll
      for (int l = 0; l < NL; ++l)
        if (l < count) {
#pragma unroll
          for (int t = 0; t < CW; ++t)
            if (c + t < n) out[(int64_t)l * n + c + t] = (double)acc[l][t];
        }
    }
    return;
  }
#pragma unroll
  for (int l4 = 0; l4 < NL / 4; ++l4) {
    if (4 * l4 >= count) break;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int t = 0; t < CW; ++t) S.red[q * CW + t][threadIdx.x] = acc[4 * l4 + q][t];
    __syncthreads();
    // the groups' sums in order: (lambda, column) pairs over all threads
    for (int idx = threadIdx.x; idx < 4 * CW * cg; idx += kAtuThreads) {
      const int v = idx / cg, k = idx % cg, l = 4 * l4 + v / CW;
      const int64_t cc = c0 + (int64_t)CW * k + v % CW;
      if (l < count && cc < n) {
        float t = S.red[v][k];
        for (int q = 1; q < rg; ++q) t += S.red[v][k + q * cg];
        out[(int64_t)l * n + cc] = (double)t;
      }
    }
  }
}

}  // namespace lmb
}  // namespace tk

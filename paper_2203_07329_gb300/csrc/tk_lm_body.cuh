// Device bodies of the float32 LSQR products for at most 16 lambda, shared by
// the single-problem kernels (tk_lm.cu) and the grouped engine (tk_group.cu).
// Both read the float32 A once in 16-byte vectors along its rows and keep the
// lambda-side operand on chip:
//  * aw_rows: store(l, i, sum_k W[l][k] A[i][k]) for the groups of ROWS rows
//    g_first, g_first + g_stride, ... < g_end, one warp per group at a time; W
//    (zero-padded to NL x n_pad) is in shared memory (load_w) by pairs of lambda,
//    so that one instruction does both multiply-adds; each lane takes 4
//    consecutive k of every 128, the next 128 loaded while the current ones are
//    used; the ROWS NL dot products per lane are added across the warp by
//    halving exchanges (each step keeps half of the values and adds the
//    partner's other half), then written.  Shared-memory reads of W (512 bytes
//    per lambda, group of rows and 128 columns) and the issue of the
//    multiply-adds bound it, not the reads of A: 262144 x 2048 with 16 / 4 lambda,
//    rows 4 / 8, 741 / 397 us one multiply-add at a time, now 581 / 347 (3.7 / 6.2 TB/s).
//  * atu_cols: out[l][c] = sum over rows rb <= i < re of U[l][i] A[i][c] for the
//    block's columns, CW per thread (NL x CW accumulators, 8 rows' loads in flight);
//    a block with fewer columns than 256 CW splits its rows over groups of threads,
//    whose sums meet in shared memory; the rows' U values are staged in shared memory
//    ([row][lambda], read as broadcasts).  Every thread of the block must call it.
#pragma once
#include "tk_internal.cuh"

namespace tk {
namespace lmb {

constexpr int kRows = 4;          // rows of A per warp (aw), the grouped engine's
constexpr int kAtuThreads = 256;  // threads of an atu block
constexpr int kAtuRB = 128;       // rows of U staged at a time (atu)
constexpr int kAwSmemCap = 200 * 1024;  // W's column chunk in shared memory (aw)

// Columns of W (and A) per chunk of the aw product: the most, in 128s, whose NL x chunk floats fit
__host__ __device__ inline int64_t aw_chunk(int nl, int64_t n) {
  const int64_t fit = (int64_t)kAwSmemCap / (4 * nl) / 128 * 128;
  const int64_t n_pad = (n + 127) / 128 * 128;
  return n_pad < fit ? n_pad : fit;
}

// Two float32 multiply-adds in one instruction (each rounded as fmaf rounds it)
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// 4 consecutive floats of a row from column k (zero past `len`); vector load when allowed
__device__ __forceinline__ float4 load4(const float* __restrict__ row, int64_t k, int64_t len, bool vec) {
  if (vec && k + 3 < len) return __ldg(reinterpret_cast<const float4*>(row + k));
  float e[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) e[t] = k + t < len ? __ldg(row + k + t) : 0.f;
  return make_float4(e[0], e[1], e[2], e[3]);
}

// W[l][k] for l < count, k < n, zero elsewhere (NL x n_pad values), in the order in which the lanes of a
// warp read it: lambda pair, 128 columns, first or second half of a lane's 4 columns, lane; 16 bytes hold
// (l, l + 1) of two columns.  The caller synchronizes.
template <int NL>
__device__ __forceinline__ void load_w(float* ws, const float* __restrict__ W, int64_t ldw, int count, int64_t n,
                                       int64_t n_pad) {
  for (int64_t idx = threadIdx.x; idx < (int64_t)NL * n_pad; idx += blockDim.x) {
    const int l = (int)(idx / n_pad);
    const int64_t k = idx % n_pad;
    const int64_t block = ((int64_t)(l / 2) * n_pad + k / 128 * 128) * 2;
    ws[block + (k & 2) * 64 + (k % 128) / 4 * 4 + (k & 1) * 2 + (l & 1)] = (l < count && k < n) ? W[(int64_t)l * ldw + k] : 0.f;
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

template <int NL, int ROWS, typename Store>
__device__ __forceinline__ void aw_rows(const float* ws, int64_t n_pad, const float* __restrict__ A, int64_t lda,
                                        int64_t m, int64_t n, int count, const Store& store, bool vec,
                                        int64_t g_first, int64_t g_stride, int64_t g_end) {
  const int lane = threadIdx.x & 31;
  const int nj = (int)(n_pad / 128);
  const ulonglong2* wl = reinterpret_cast<const ulonglong2*>(ws) + lane;  // 64 of these per lambda pair and 128 columns
  for (int64_t g = g_first; g < g_end; g += g_stride) {
    const int64_t i0 = g * ROWS;
    const float* row0 = A + i0 * lda;
    const int rmax = (int)(m - i0 < ROWS ? m - i0 : ROWS);
    f32x2 acc[ROWS][NL / 2];
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
#pragma unroll
      for (int l = 0; l < NL / 2; ++l) acc[r][l] = 0;
    float4 cur[ROWS], nxt[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
      cur[r] = r < rmax ? load4(row0 + r * lda, 4 * lane, n, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
    for (int j = 0; j < nj; ++j) {
      const int64_t k = (int64_t)128 * j + 4 * lane;
      if (j + 1 < nj) {
#pragma unroll
        for (int r = 0; r < ROWS; ++r)
          nxt[r] = r < rmax ? load4(row0 + r * lda, k + 128, n, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        f32x2 a0[ROWS], a1[ROWS];  // the lane's columns 2 h and 2 h + 1, twice each
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
          a0[r] = h ? pack2(cur[r].z, cur[r].z) : pack2(cur[r].x, cur[r].x);
          a1[r] = h ? pack2(cur[r].w, cur[r].w) : pack2(cur[r].y, cur[r].y);
        }
#pragma unroll
        for (int l = 0; l < NL / 2; ++l) {
          const ulonglong2 w = wl[((int64_t)l * nj + j) * 64 + 32 * h];
#pragma unroll
          for (int r = 0; r < ROWS; ++r) acc[r][l] = fma2(a1[r], w.y, fma2(a0[r], w.x, acc[r][l]));
        }
      }
#pragma unroll
      for (int r = 0; r < ROWS; ++r) cur[r] = nxt[r];
    }
    // add the V = ROWS NL values across the warp: each halving step keeps half (the lanes with bit s
    // set keep the upper half) and adds the partner's copy of it; once one value is left, plain steps
    constexpr int V = ROWS * NL;
    float v[V];
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
#pragma unroll
      for (int l = 0; l < NL / 2; ++l) unpack2(acc[r][l], v[r * NL + 2 * l], v[r * NL + 2 * l + 1]);
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
    // lane holds values qbase .. qbase + nv - 1 (V >= 32: V / 32 per lane; V = 16: the same value on
    // two lanes, written by the one with bit 0 clear)
    const bool writer = V >= 32 || (lane & 1) == 0;
    if (writer) {
#pragma unroll
      for (int t = 0; t < (V + 31) / 32; ++t) {
        const int q = qbase + t, r = q / NL, l = q % NL;
        const int64_t i = i0 + r;
        if (i < m && l < count) store(l, i, v[t]);
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

// The block's columns c0 .. c0 + width - 1 (those < n; width a multiple of 32 CW, at most CW kAtuThreads), rows rb .. re - 1.  CW columns per
// thread (4 for <= 8 lambda, 2 for 16: NL x CW accumulators), 8 rows' loads in flight.
template <int NL, int CW>
__device__ __forceinline__ void atu_cols(AtuSmem<NL, CW>& S, const float* __restrict__ A, int64_t lda, int64_t n,
                                         const float* __restrict__ U, int64_t ldu, int count, int64_t rb, int64_t re,
                                         int64_t c0, int width, double* __restrict__ out, bool vec) {
  // cg threads across the columns (whole warps), rg groups of rows
  const int64_t cols = n - c0 < width ? n - c0 : width;
  const int cg = (int)((cols + 32 * CW - 1) / (32 * CW)) * 32, rg = kAtuThreads / cg;
  const int g = threadIdx.x / cg;
  const int64_t c = g < rg ? c0 + (int64_t)CW * (threadIdx.x % cg) : n;
  constexpr int RU = 8;
  // Up to 8 lambda: lambda pairs, two multiply-adds per instruction (4 lambda, 262144 x 2048: 395 -> 305 us;
  // 8 lambda: 552 -> 376).  With 16 lambda x 2 columns the pairs' moves cost what they save (583 us, 620 in
  // pairs): one by one.
  constexpr bool PAIRS = NL <= 8;
  f32x2 acc[PAIRS ? NL / 2 : 1][CW];
  float sum[NL][CW];
#pragma unroll
  for (int l = 0; l < (PAIRS ? NL / 2 : 1); ++l)
#pragma unroll
    for (int t = 0; t < CW; ++t) acc[l][t] = 0;
#pragma unroll
  for (int l = 0; l < NL; ++l)
#pragma unroll
    for (int t = 0; t < CW; ++t) sum[l][t] = 0.f;
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
          if constexpr (PAIRS) {
            f32x2 ad[CW];
#pragma unroll
            for (int t = 0; t < CW; ++t) ad[t] = pack2(a[q][t], a[q][t]);
#pragma unroll
            for (int l4 = 0; l4 < NL / 4; ++l4) {
              const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(&S.us[r + q][4 * l4]);
#pragma unroll
              for (int t = 0; t < CW; ++t) {
                acc[2 * l4][t] = fma2(u.x, ad[t], acc[2 * l4][t]);
                acc[2 * l4 + 1][t] = fma2(u.y, ad[t], acc[2 * l4 + 1][t]);
              }
            }
          } else {
#pragma unroll
            for (int l4 = 0; l4 < NL / 4; ++l4) {
              const float4 u4 = *reinterpret_cast<const float4*>(&S.us[r + q][4 * l4]);
              const float uu[4] = {u4.x, u4.y, u4.z, u4.w};
#pragma unroll
              for (int t4 = 0; t4 < 4; ++t4)
#pragma unroll
                for (int t = 0; t < CW; ++t) sum[4 * l4 + t4][t] = fmaf(uu[t4], a[q][t], sum[4 * l4 + t4][t]);
            }
          }
        }
      }
    }
  }
  if constexpr (PAIRS) {
#pragma unroll
    for (int l = 0; l < NL / 2; ++l)
#pragma unroll
      for (int t = 0; t < CW; ++t) unpack2(acc[l][t], sum[2 * l][t], sum[2 * l + 1][t]);
  }
  if (rg == 1) {
    if (c < n) {
#pragma unroll
      for (int l = 0; l < NL; ++l)
        if (l < count) {
#pragma unroll
          for (int t = 0; t < CW; ++t)
            if (c + t < n) out[(int64_t)l * n + c + t] = (double)sum[l][t];
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
      for (int t = 0; t < CW; ++t) S.red[q * CW + t][threadIdx.x] = sum[4 * l4 + q][t];
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

// Float64-accurate products on the BF16 tensor cores (splitting into exact
// integer slices, in the manner of Ozaki's error-free matrix multiplication).
//
// GB300 issues about two float64 FMA per clock per SM, so float64 products
// (the Gram matrix, the Cholesky trailing updates, the refinement's r = b - X A^T
// and A^T r, and the LSQR products of the float64 form) are bound by that pipe:
// one product of 65536 x 1024 with 16 lambda takes 3.8 ms there and 0.25 ms from
// digits.  Here every row of an operand is scaled by a power of two 2^E (E one
// above the exponent of its largest entry, so that 2^(E-2) <= max |x| < 2^(E-1);
// A is scaled along its columns first, see k_oz_scale_slice), rounded to
// nearest at 2^(E-57) (within 2^-55 of the row maximum) and written with
// S = 8 balanced base-128 digits,
//   x 2^-E = sum_p d_p 2^(-7(p+1)),  d_p in [-64, 64],
// taken from the least significant end with carries; each digit is exact in
// BF16.  A product of two digits is an integer of magnitude <= 2^12; the pairs
// (p, q) with p + q = t share one FP32 accumulator ("level" t), and a level
// sum of at most 8 pairs over 256 values of K stays below 2^24, so the tensor
// core's FP32 accumulation is exact.  Every 256 values of K the level sums
// are added, with their weights 2^(-7(t+2)), exactly into two int64
// accumulators per output (levels 0-3 and 4-7), made one double at the
// end (with 4 digits: scaled into FP32 accumulators).  The 28
// pairs with p + q > 7 are dropped: at most 7.1 * 2^-58 of 2^(Ea+Ex), i.e.
// 2^-51 of max|a| max|x| per product when every digit is +-64 (typical digits
// give far less).  The result carries errors of a few float64 units relative
// to the row maxima: the normwise accuracy of a float64 GEMM (the tests check
// it element by element against extended-precision products).  Cut after 4
// digits, the same slices are a round-to-nearest 28-bit representation.
//
// The products run on tcgen05 (kind::f16, M = 128, K = 16; per digit p of the
// big operand one MMA of N = 32 (S - p) over the stacked digit planes of the
// small one), operands brought in by TMA in the 128-byte swizzle layout, the
// level accumulators in tensor memory, double-buffered so that four epilogue
// warps flush one 256-value chunk of K while the MMAs of the next chunk run.
#include <algorithm>
#include <climits>
#include <type_traits>
#include <cuda_bf16.h>

#include "tk_internal.cuh"
#include "tk_tcgen05.cuh"

namespace tk {
namespace {

constexpr int OZ_S = 8;          // slices
constexpr int OZ_LV = OZ_S;      // levels t = p + q in 0..7 kept
constexpr int OZ_KPAD = 64;      // slice rows are padded to a multiple of 64 values of K (one TMA box)

// Exponent marking a row or column with an inf or NaN: its digits are zero
// and every output that uses it is NaN, so non-finite input is reported (the
// LSQR stop tests and the refinement see it) instead of being dropped.
// A marked exponent is OZ_EBAD plus the exponent of the finite entries (0 for a column), which the
// digits of those entries use.
constexpr int OZ_EBAD = 1 << 24;
__host__ __device__ constexpr bool oz_bad(int e) { return e > OZ_EBAD / 2; }
__host__ __device__ constexpr int oz_val(int e) { return oz_bad(e) ? e - OZ_EBAD : e; }
// Exponent of a row that holds only zeros so far (a memset pattern; far below every exponent, and
// adding any exponent to it does not overflow).
constexpr int OZ_EZERO = (int)0x80808080;

// max(m, |x|) that turns inf and NaN into +inf (fmax would ignore a NaN).
__device__ __forceinline__ double oz_absmax(double m, double x) {
  const double a = fabs(x);
  return a <= m ? m : (a == a ? a : __longlong_as_double(0x7ff0000000000000ll));
}
// The exponent of a maximum: one above frexp's (0 for 0, OZ_EBAD if not finite).
__device__ __forceinline__ int oz_exponent(double mx) {
  if (!(mx <= 1.7976931348623157e308)) return OZ_EBAD;
  int e = 0;
  if (mx > 0.0) {
    frexp(mx, &e);  // mx = f 2^e, 0.5 <= f < 1
    ++e;            // so mx < 2^(e-1)
  }
  return e;
}

// One above frexp's exponent of x, from the bit pattern: 2^(E-2) <= |x| < 2^(E-1) (OZ_EZERO for 0).
// *bad is set for inf and NaN, which count as 0.
__device__ __forceinline__ int oz_exp_of(double x, bool* bad) {
  const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
  if (ex == 0x7ff) {
    *bad = true;
    return OZ_EZERO;
  }
  if (ex) return ex - 1021;
  const long long mant = __double_as_longlong(x) & ((1ll << 52) - 1);
  return mant ? (63 - __clzll(mant)) - 1072 : OZ_EZERO;
}
__device__ __forceinline__ int oz_exp_of(float x, bool* bad) {
  const int b = __float_as_int(x), ex = (b >> 23) & 0xff;
  if (ex == 0xff) {
    *bad = true;
    return OZ_EZERO;
  }
  if (ex) return ex - 125;
  const int mant = b & 0x7fffff;
  return mant ? (31 - __clz(mant)) - 147 : OZ_EZERO;
}

// Exponent E with max_r |X[r][c]| < 2^(E-1) per column (0 for a zero column):
// the bit patterns of non-negative doubles order like the values, so the
// column maxima are combined with an integer atomicMax (mx zeroed first).
// With copy != nullptr the same pass writes the float32 copy of X (row stride cols) that the
// float32 products read: A crosses HBM once for both.
template <typename T>
__global__ void __launch_bounds__(256) k_oz_colmax(const T* __restrict__ X, int64_t rows, int64_t cols, int64_t ld,
                                                   int64_t rows_per, unsigned long long* __restrict__ mx,
                                                   float* __restrict__ copy) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cols) return;
  const int64_t r0 = (int64_t)blockIdx.y * rows_per, r1 = r0 + rows_per < rows ? r0 + rows_per : rows;
  double v = 0.0;
  int64_t r = r0;
  for (; r + 8 <= r1; r += 8) {
    T x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = X[(r + k) * ld + c];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      v = oz_absmax(v, (double)x[k]);
      if (copy) copy[(r + k) * cols + c] = (float)x[k];
    }
  }
  for (; r < r1; ++r) {
    const T x = X[r * ld + c];
    v = oz_absmax(v, (double)x);
    if (copy) copy[r * cols + c] = (float)x;
  }
  atomicMax(&mx[c], (unsigned long long)__double_as_longlong(v));  // +inf orders above every finite value
}
__global__ void k_oz_colexp(const unsigned long long* __restrict__ mx, int64_t cols, int* __restrict__ E) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cols) return;
  E[c] = oz_exponent(__longlong_as_double((long long)mx[c]));
}

// round(x 2^(56-E)) (|x 2^-E| < 1/2, so |result| <= 2^55) from the bit
// pattern of x: no float64 instruction (GB300 issues those at a fraction of
// the integer rate).  Ties round away from zero.
__device__ __forceinline__ long long oz_fixed(double x, int E) {
  const long long bits = __double_as_longlong(x);
  int ex = (int)((bits >> 52) & 0x7ff);
  long long mant = bits & ((1ll << 52) - 1);
  if (ex) mant |= 1ll << 52;
  else ex = 1;  // subnormal: same scale as the smallest normal exponent
  const int sh = ex - 1019 - E;  // |x| 2^(56-E) = mant 2^sh
  long long u;
  if (sh >= 0) u = mant << sh;  // mant 2^sh < 2^55: sh < 55
  else if (sh > -63) u = (mant + (1ll << (-sh - 1))) >> (-sh);
  else u = 0;
  return bits < 0 ? -u : u;
}
__device__ __forceinline__ long long oz_fixed(float x, int E) {
  const int bits = __float_as_int(x);
  int ex = (bits >> 23) & 0xff;
  long long mant = bits & 0x7fffff;
  if (ex) mant |= 0x800000;
  else ex = 1;
  const int sh = ex - 94 - E;  // |x| 2^(56-E) = mant 2^sh
  long long u;
  if (sh >= 0) u = mant << sh;  // mant 2^sh < 2^55: sh < 55 (subnormal x: small mant)
  else if (sh > -63) u = (mant + (1ll << (-sh - 1))) >> (-sh);
  else u = 0;
  return bits < 0 ? -u : u;
}

// BF16 bits of a small integer (|d| <= 2^8): through the float with the
// 1.5 * 2^23 offset; its low 16 bits are zero, so the top half is exact.
__device__ __forceinline__ unsigned short oz_bf16_bits(int d) {
  const float f = __int_as_float(0x4B400000 + d) - 12582912.0f;
  return (unsigned short)(__float_as_uint(f) >> 16);
}

// The 8 balanced base-128 digits of v (|v| <= 2^55): d = ((u + 64) mod 128)
// - 64 from the bottom, carry (u - d) / 128, on two 32-bit halves (the low 28
// bits, then the rest plus the carry); the last carry is the top digit,
// |d_0| <= 64.  bits[p] = BF16 bit pattern of d_p.
__device__ __forceinline__ void oz_digits(long long v, unsigned short (&bits)[OZ_S]) {
  int lo = (int)(v & ((1ll << 28) - 1));
  int hi = (int)(v >> 28);
#pragma unroll
  for (int p = OZ_S - 1; p >= 4; --p) {
    const int d = ((lo + 64) & 127) - 64;
    bits[p] = oz_bf16_bits(d);
    lo = (lo - d) >> 7;
  }
  hi += lo;
#pragma unroll
  for (int p = 3; p >= 1; --p) {
    const int d = ((hi + 64) & 127) - 64;
    bits[p] = oz_bf16_bits(d);
    hi = (hi - d) >> 7;
  }
  bits[0] = oz_bf16_bits(hi);
}

// x, or 0 for inf and NaN (their row or column is marked)
__device__ __forceinline__ double oz_finite(double x) {
  return ((__double2hiint(x) >> 20) & 0x7ff) == 0x7ff ? 0.0 : x;
}
__device__ __forceinline__ float oz_finite(float x) { return ((__float_as_int(x) >> 23) & 0xff) == 0xff ? 0.f : x; }

template <typename T>
__device__ __forceinline__ void oz_split(T x, int E, unsigned short (&bits)[OZ_S]) {
  oz_digits(oz_fixed(x, E), bits);
}
__device__ __forceinline__ unsigned oz_pack(unsigned short a, unsigned short b) { return (unsigned)a | ((unsigned)b << 16); }

// Row exponents and digit planes of a matrix A (rows x cols, row stride ld) whose columns are scaled
// by 2^-EC: with A'' = A[r][c] 2^-(ER[r] + EC[c]), ER the smallest exponents with |A''| < 1/2, planes
// out[p][r][c] (row stride cols_pad, zero in the padding) with A'' = sum_p out[p][r][c] 2^(-7(p+1)) to
// within 2^-57.  Scaling the columns first makes the digits independent of the columns' units, and
// lets one set of planes serve both products: A W^T reads it along the rows (K = columns), A^T U
// along the columns (K = rows, the operand MN-major).
// A block owns a band of RB rows: its 8 warps find the RB exponents (8 / RB warps to a row), then
// all threads split the band, whose second read comes from L2 (RB is chosen so that the bands of the
// resident blocks fit there).  Bound by HBM: one read of A and 16 bytes written per element; 262144 x
// 2048 float64 takes 3.0 ms (and 1.1 ms for the column maxima and the float32 copy) where separate row
// and column planes took 9.5 ms.
template <typename T>
__global__ void __launch_bounds__(256) k_oz_scale_slice(const T* __restrict__ A, int64_t rows, int64_t cols,
                                                        int64_t ld, const int* __restrict__ EC, int RB,
                                                        int64_t cols_pad, int* __restrict__ ER,
                                                        __nv_bfloat16* __restrict__ out) {
  __shared__ int sh_e[8], sh_bad[8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t r0 = (int64_t)blockIdx.x * RB;
  const int nr = rows - r0 < RB ? (int)(rows - r0) : RB;
  if (threadIdx.x < 8) {
    sh_e[threadIdx.x] = OZ_EZERO;
    sh_bad[threadIdx.x] = 0;
  }
  __syncthreads();
  const int wpr = 8 / RB;  // warps to a row
  const int lr = warp / wpr;
  if (lr < nr) {
    const T* x = A + (r0 + lr) * ld;
    int e = OZ_EZERO;
    bool bad = false;
#pragma unroll 8
    for (int64_t c = (warp % wpr) * 32 + lane; c < cols; c += wpr * 32) {
      const int ex = oz_exp_of(x[c], &bad);
      const int ec = oz_val(EC[c]);
      e = max(e, ex == OZ_EZERO ? OZ_EZERO : ex - ec);
    }
    e = __reduce_max_sync(0xffffffffu, e);
    bad = __any_sync(0xffffffffu, bad);
    if (lane == 0) {
      atomicMax(&sh_e[lr], e);
      if (bad) sh_bad[lr] = 1;
    }
  }
  __syncthreads();
  if (threadIdx.x < nr) {
    const int e = sh_e[threadIdx.x] == OZ_EZERO ? 0 : sh_e[threadIdx.x];
    ER[r0 + threadIdx.x] = e + (sh_bad[threadIdx.x] ? OZ_EBAD : 0);
    sh_e[threadIdx.x] = e;
  }
  __syncthreads();
  const int64_t plane = rows * cols_pad;
  for (int64_t c = 2 * threadIdx.x; c < cols_pad; c += 2 * blockDim.x) {
    const int e0 = c < cols ? oz_val(EC[c]) : 0, e1 = c + 1 < cols ? oz_val(EC[c + 1]) : 0;
    for (int k = 0; k < nr; ++k) {
      const T* x = A + (r0 + k) * ld;
      const int e = sh_e[k];
      unsigned short s0[OZ_S], s1[OZ_S];
      oz_split(c < cols ? oz_finite(x[c]) : T(0), e + e0, s0);
      oz_split(c + 1 < cols ? oz_finite(x[c + 1]) : T(0), e + e1, s1);
      unsigned* o = reinterpret_cast<unsigned*>(out + (r0 + k) * cols_pad + c);
#pragma unroll
      for (int p = 0; p < OZ_S; ++p) o[p * (plane / 2)] = oz_pack(s0[p], s1[p]);
    }
  }
}

// Digits of the lambda rows of a vector block V (M x K, row stride ld), the small operand of a
// product: with V'[l][k] = V[l][k] 2^shift[k] (shift: the exponents of A that the product sums over;
// null = 0), E[l] one above the exponent of the row's largest |V'| and planes out[p][l][k] (row
// stride kp, zero in the padding).  Rows of fewer than OZ_VEC_LONG values: one block per row does
// both (the row comes from L1 or L2 the second time); longer rows: the exponents by blocks of
// values (k_oz_vec_exp, E preset to OZ_EZERO by a memset), then k_oz_vec_slice.
constexpr int64_t OZ_VEC_LONG = 8192;
template <typename T>
__device__ __forceinline__ int oz_vec_exp(const T* __restrict__ x, const int* __restrict__ shift, int64_t k0,
                                          int64_t k1, bool* bad) {
  int e = OZ_EZERO;
#pragma unroll 4
  for (int64_t k = k0 + threadIdx.x; k < k1; k += blockDim.x) {
    const int ex = oz_exp_of(x[k], bad);
    const int sk = shift ? oz_val(shift[k]) : 0;
    e = max(e, ex == OZ_EZERO ? OZ_EZERO : ex + sk);
  }
  return e;
}
// max over the block; a non-finite value anywhere marks it
__device__ __forceinline__ int oz_block_exp(int e, bool bad, int* sh) {
  e = __reduce_max_sync(0xffffffffu, bad ? OZ_EBAD : e);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = e;
  __syncthreads();
  e = sh[0];
  for (int w = 1; w < (int)(blockDim.x >> 5); ++w) e = max(e, sh[w]);
  return e;
}
template <typename T>
__device__ __forceinline__ void oz_vec_split(const T* __restrict__ x, const int* __restrict__ shift, int64_t k,
                                             int64_t K, int e, int64_t plane, int planes, unsigned* __restrict__ o) {
  // a marked row's digits are not used (every output of it is NaN); a zero row has zero digits
  const bool none = oz_bad(e) || e == OZ_EZERO;
  unsigned short s0[OZ_S], s1[OZ_S];
  oz_split(k < K && !none ? x[k] : T(0), (none || !shift || k >= K) ? (none ? 0 : e) : e - oz_val(shift[k]), s0);
  oz_split(k + 1 < K && !none ? x[k + 1] : T(0),
           (none || !shift || k + 1 >= K) ? (none ? 0 : e) : e - oz_val(shift[k + 1]), s1);
#pragma unroll
  for (int p = 0; p < OZ_S; ++p)
    if (p < planes) o[p * (plane / 2)] = oz_pack(s0[p], s1[p]);
}
template <typename T>
__global__ void __launch_bounds__(512) k_oz_vec(const T* __restrict__ V, int64_t M, int64_t K, int64_t ld,
                                                const int* __restrict__ shift, int* __restrict__ E, int64_t kp,
                                                int planes, __nv_bfloat16* __restrict__ out) {
  __shared__ int sh[16];
  const int64_t l = blockIdx.x;
  const T* x = V + l * ld;
  bool bad = false;
  int e = oz_vec_exp(x, shift, 0, K, &bad);
  e = oz_block_exp(e, bad, sh);
  if (threadIdx.x == 0) E[l] = e;
  for (int64_t k = 2 * threadIdx.x; k < kp; k += 2 * blockDim.x)
    oz_vec_split(x, shift, k, K, e, M * kp, planes, reinterpret_cast<unsigned*>(out + l * kp + k));
}
template <typename T>
__global__ void __launch_bounds__(256) k_oz_vec_exp(const T* __restrict__ V, int64_t K, int64_t ld,
                                                    const int* __restrict__ shift, int64_t per_block,
                                                    int* __restrict__ E) {
  __shared__ int sh[8];
  const int64_t k0 = (int64_t)blockIdx.x * per_block;
  const int64_t k1 = k0 + per_block < K ? k0 + per_block : K;
  bool bad = false;
  int e = oz_vec_exp(V + (int64_t)blockIdx.y * ld, shift, k0, k1, &bad);
  e = oz_block_exp(e, bad, sh);
  if (threadIdx.x == 0) atomicMax(&E[blockIdx.y], e);  // OZ_EBAD wins
}
template <typename T>
__global__ void __launch_bounds__(256) k_oz_vec_slice(const T* __restrict__ V, int64_t M, int64_t K, int64_t ld,
                                                      const int* __restrict__ shift, const int* __restrict__ E,
                                                      int64_t kp, int planes, __nv_bfloat16* __restrict__ out) {
  const int64_t l = blockIdx.y;
  const int e = E[l];
  const int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 2;
  if (k < kp) oz_vec_split(V + l * ld, shift, k, K, e, M * kp, planes, reinterpret_cast<unsigned*>(out + l * kp + k));
}

// Slices of the COLUMNS of X (rows x cols) with column exponents E, stored
// transposed: planes out[p][c][r] (row stride rows_pad, zero in the padding).
// 64 x 32 tiles through shared memory: reads of 32 consecutive columns, and
// per plane 128-byte stores of 64 consecutive rows (two per thread); grid.x
// runs over row tiles, grid.y over column tiles.
template <typename T>
__global__ void __launch_bounds__(256) k_oz_slice_t(const T* __restrict__ X, int64_t rows, int64_t cols, int64_t ld,
                                                    const int* __restrict__ E, int64_t rows_pad,
                                                    __nv_bfloat16* __restrict__ out) {
  __shared__ T tile[64][33];
  const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
  const int64_t r0 = (int64_t)blockIdx.x * 64, c0 = (int64_t)blockIdx.y * 32;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int64_t r = r0 + ty + 8 * i, c = c0 + tx;
    tile[ty + 8 * i][tx] = (r < rows && c < cols) ? X[r * ld + c] : T(0);
  }
  __syncthreads();
  const int64_t plane = cols * rows_pad;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int cc = ty + 8 * i;
    const int64_t c = c0 + cc, r = r0 + 2 * tx;
    if (c < cols && r < rows_pad) {  // rows_pad is a multiple of 64: r + 1 < rows_pad too
      const int e = E[c];
      unsigned short s0[OZ_S], s1[OZ_S];
      oz_split(tile[2 * tx][cc], e, s0);
      oz_split(tile[2 * tx + 1][cc], e, s1);
      unsigned* o = reinterpret_cast<unsigned*>(out + c * rows_pad + r);
#pragma unroll
      for (int p = 0; p < OZ_S; ++p) o[p * (plane / 2)] = oz_pack(s0[p], s1[p]);
    }
  }
}

// ---- the product on tcgen05 ---------------------------------------------------
// D[r][l] = sum_k P[r][k] Q[l][k] from the first S digit planes of P (rows x
// K, row exponents EP) and of Q (M x K, row exponents EQ), Q K-major.  P is
// K-major (TR = false: the planes hold P row by row) or MN-major (TR = true:
// the planes hold P^T, K rows of `rows` values; the A^T products read the
// planes of A this way, two boxes of 64 K x 64 rows of P per ring slot).
// S = 8: float64 accuracy (levels added exactly into int64 accumulators, one
// rounding at the end); S = 4: the 28-bit rounded operands, float32 accuracy
// (levels flushed into float32).
// Tile: 128 rows of P x 32 (64) rows of Q x one K split.  A CTA per slot of the GPU runs through its tiles
// with the rings and tensor-memory buffers going on from one to the next, so the last step of a tile (float64
// arithmetic, reads of U) overlaps the products of the next (a CTA per tile: 4 digits, 64 lambda, 262144 x 4096
// 1.85 ms, now 1.44 = 5.9 TB/s of planes; 32 lambda, 262144 x 2048 0.75, now 0.65; 8 digits, 65536 x 1024, 16
// lambda 235 us, now 201, of which a quarter of the last of 3.4 rounds of tiles is idle).
//   warp 0 (one lane): TMA producer -- per 64 values of K the S planes of Q
//     (4 KiB each) into a 2-slot ring, then the S planes of P one by one
//     (16 KiB each) into an 8-slot ring;
//   warp 1 (one lane): MMA issuer -- for plane p of P, D_(p+q) += P_p Q_q^T
//     for every q <= S-1-p as one MMA of N = 32 (S - p) (4 of K = 16); the
//     level accumulators of a chunk of 256 values of K sit in one of two
//     tensor-memory buffers;
//   warp 2: allocates / frees the 2 S 32 tensor-memory columns;
//   warps 4-7: epilogue -- per chunk, read the S levels (lanes 32(w-4) ..),
//     add them into 32 accumulators per row, release the buffer; at the end
//     write the result: MODE 0 R[l][r] = b[r] - D (float64); MODE 1
//     partial[z][l][r] = D (float64); MODE 2 U[l][r] = D + coef[l] U[l][r]
//     (coef == nullptr: U = D; U float32 for S = 4, float64 for S = 8).
// Every mbarrier wait is bounded; a wait that gives up sets *err and the
// roles stop.
constexpr int OT_M = 128;
constexpr int OT_N = 32;
constexpr int OT_KB = 64;
constexpr int OT_CHUNK = 256;
constexpr int OT_KB_PER_CHUNK = OT_CHUNK / OT_KB;
constexpr int64_t OT_MAX_KPS = int64_t(1) << 27;  // values of K per split that the int64 level sums hold exactly
constexpr uint32_t OT_P_BYTES = OT_M * OT_KB * 2;   // 16 KiB

// CTA shapes (tensor memory: 2 buffers x S levels x NT columns <= 512):
//   S = 8, NT = 32 (float64-accurate passes): one CTA per SM, an 8-slot ring of P planes;
//   S = 4, NT = 32 (float32 LSQR products, <= 32 lambda): 4 slots and 256 columns, so two
//     CTAs share an SM and one streams while the other starts up or flushes its last chunk;
//   S = 4, NT = 64 (more than 32 lambda): one CTA per SM over 64 lambda, so the digit planes
//     of the big operand are read once for 64 lambda instead of once per 32.
template <int S, int NT>
struct OtCfg {
  static constexpr bool WIDE = S == OZ_S || NT == 64;
  static constexpr int PST = WIDE ? 8 : 4;
  static constexpr int CTAS_PER_SM = WIDE ? 1 : 2;
  static constexpr uint32_t QS_BYTES = NT * OT_KB * 2;  // one digit plane of the small operand
};

template <int S, int NT>
struct OtSmem {
  static constexpr int PST = OtCfg<S, NT>::PST;
  uint8_t p[PST][OT_P_BYTES];
  uint8_t q[2][S * OtCfg<S, NT>::QS_BYTES];
  uint64_t p_full[PST];
  uint64_t p_empty[PST];
  uint64_t q_full[2];
  uint64_t q_empty[2];
  uint64_t acc_full[2];
  uint64_t acc_empty[2];
  uint64_t mma_drain;  // error path: completes when every MMA the CTA issued is done
  uint32_t tmem_base;
};

// MODE 3: many h x h products (h a multiple of 128), the blocks of a level of the triangular inverse:
// batch z = (matrix, pair) holds rows z h .. z h + h - 1 of both operands' planes (K = h);
// out[z / pairs * mstride + z % pairs * pstride + l ldo + r] = sign D, float64 (S = 8) or float32 (S = 4),
// for l < min(h, n - (2 pair + 1) h).  Triangular operands skip the K they hold zeros in: tri 1: Q's row l
// ends at k = l; tri 2: P's row r starts at k = r.
struct OtTri {
  int pairs, tri, h, n;
  int64_t mstride, pstride;
  double sign;
};

// 2^e as a double (e within the normal range).
__device__ __forceinline__ double pow2d(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }

// v 2^s as a double, built from the integer's bits with integer instructions
// only (GB300's float64 pipe is the bottleneck of the update's epilogue):
// exact for |v| < 2^53.  *ok = false when the result would not be a normal
// double (the caller then takes the float64 route).
__device__ __forceinline__ double i53_scaled(long long v, int s, bool* ok) {
  if (v == 0) return 0.0;
  const unsigned long long sg = v < 0 ? (1ull << 63) : 0ull;
  const unsigned long long a = v < 0 ? (unsigned long long)(-v) : (unsigned long long)v;
  const int p = 63 - __clzll((long long)a);  // a in [2^p, 2^(p+1)), p <= 52
  const int ex = p + s + 1023;
  if (ex < 1 || ex > 2046) {
    *ok = false;
    return 0.0;
  }
  const unsigned long long mant = (a << (52 - p)) & ((1ull << 52) - 1);
  return __longlong_as_double((long long)(sg | ((unsigned long long)ex << 52) | mant));
}

struct OtTiles {
  uint32_t gx, gy, gz;
};

// Threads of the result's warps.  MODE 4 has one chunk of products per tile, so reading a tile's sums out of
// tensor memory and scaling them into T takes longer than the products: 8 warps (order 4096, 64 lambda: 4 warps,
// each with its 32 columns' sums in registers and T read behind them, 4.35 ms a panel on average, now 3.39).
template <int MODE>
constexpr int ot_epi = MODE == 4 ? 256 : 128;

// MODE 4: the trailing update of a Cholesky panel of 256 rows, for every lambda: T[l][r] -= D for r >= l, T the
// w x w trailing block (rows ldo apart, lambda z at out + z mstride), P = Q = the panel's planes (lambda z's
// columns at rows z h; K = 256).  Tiles: the blocks of 128 x 128 on and above the diagonal, 4 tiles of 32 each.

// SYM: a symmetric product (P = Q), of which out[l][r] is wanted for l <= r only, by a CTA per tile: the hardware's own
// order shares out the tiles, half of which leave before they set anything up, better than CTAs that run through
// them, and the row tiles of a column of tiles follow one another (the Gram matrix, bound by the products:
// 8192 x 2048 1.54 ms with the rotated order and the skipped tiles' setup, now 1.40; 8192 x 4096 5.05, now 4.59).
template <int S, int MODE, int NT, bool TR, bool SYM>
__global__ void __launch_bounds__(128 + ot_epi<MODE>, OtCfg<S, NT>::CTAS_PER_SM)
    k_oz_tc(const __grid_constant__ CUtensorMap tmP, const __grid_constant__ CUtensorMap tmQ,
            const int* __restrict__ EP, const int* __restrict__ EQ, int64_t rows, int M, int64_t K, int64_t kps,
            const double* __restrict__ b, void* __restrict__ out, int64_t ldo, const double* __restrict__ coef,
            int* __restrict__ err, const OtTiles tiles, const OtTri tri) {
  using Acc = typename std::conditional<S == OZ_S, double, float>::type;
  constexpr uint32_t TMEM_COLS = 2 * S * NT;
  constexpr uint32_t QS_BYTES = OtCfg<S, NT>::QS_BYTES;
  constexpr uint32_t Q_BYTES = S * QS_BYTES;
  extern __shared__ __align__(1024) uint8_t ot_raw[];
  OtSmem<S, NT>& Sm = *reinterpret_cast<OtSmem<S, NT>*>((reinterpret_cast<uintptr_t>(ot_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Tile t of the launch: gx row tiles x gy column tiles x gz splits (MODE 3: batches); false: nothing to do.
  struct Tile {
    int64_t r0, kbeg;
    int l0, z, M, prow, nkb, nch;  // prow: first row of the batch in the operands' planes and exponents
  };
  const auto tile_at = [&](uint32_t t, Tile& T) -> bool {
    uint32_t x = t, y = 0;
    T.z = 0;
    if constexpr (MODE == 4) {
      const uint32_t per = tiles.gx, q = t / per, b = (t - q * per) / 4;
      T.z = (int)q;
      x = (uint32_t)((sqrtf(8.f * (float)b + 1.f) - 1.f) * 0.5f);
      while (x * (x + 1) / 2 > b) --x;
      while ((x + 1) * (x + 2) / 2 <= b) ++x;
      y = 4 * (b - x * (x + 1) / 2) + t % 4;  // (per is a multiple of 4)
    } else if (t >= tiles.gx) {
      // the row tile rotates with q: with gx a divisor of the grid a CTA would otherwise keep one row tile, and
      // where the work of a tile depends on it (MODE 3) the CTAs would end up unequal
      const uint32_t q = t / tiles.gx;
      x = SYM ? t - q * tiles.gx : (t - q * tiles.gx + q) % tiles.gx;
      y = q % tiles.gy;
      T.z = (int)(q / tiles.gy);
    }
    T.r0 = (int64_t)x * OT_M;
    T.l0 = (int)y * NT;
    T.M = M;
    T.prow = 0;
    if (SYM && T.l0 > T.r0 + OT_M - 1) return false;
    int64_t kend;
    if constexpr (MODE == 3) {
      const int left = tri.n - (2 * (T.z % tri.pairs) + 1) * tri.h;
      T.M = left < tri.h ? left : tri.h;
      if (T.l0 >= T.M) return false;
      T.prow = T.z * tri.h;
      T.kbeg = tri.tri == 2 ? T.r0 : 0;
      kend = tri.tri == 1 && T.l0 + NT < K ? T.l0 + NT : K;
    } else if constexpr (MODE == 4) {
      if (T.l0 >= M) return false;
      T.prow = T.z * tri.h;
      T.kbeg = 0;
      kend = K;
    } else {
      T.kbeg = (int64_t)T.z * kps;
      kend = K < T.kbeg + kps ? K : T.kbeg + kps;
    }
    T.nkb = kend > T.kbeg ? (int)((kend - T.kbeg + OT_KB - 1) / OT_KB) : 0;
    T.nch = (T.nkb + OT_KB_PER_CHUNK - 1) / OT_KB_PER_CHUNK;
    return true;
  };
  const uint32_t ntiles = tiles.gx * tiles.gy * tiles.gz;
  Tile T;  // the first tile, found while the barriers and tensor memory are set up
  bool has = tile_at(blockIdx.x, T);
  if (SYM && !has) return;
  // the CTA's next tile
  const auto next_tile = [&](uint32_t& t) {
    t = SYM ? ntiles : t + gridDim.x;
    has = t < ntiles && tile_at(t, T);
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < OtCfg<S, NT>::PST; ++s) {
      mbar_init(&Sm.p_full[s], 1);
      mbar_init(&Sm.p_empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&Sm.q_full[s], 1);
      mbar_init(&Sm.q_empty[s], 1);
      mbar_init(&Sm.acc_full[s], 1);
      mbar_init(&Sm.acc_empty[s], ot_epi<MODE>);
    }
    mbar_init(&Sm.mma_drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&Sm.tmem_base)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = Sm.tmem_base;

  if (warp == 0 && lane == 0) {
    uint32_t g = 0, gq = 0;  // loads issued into the P ring and the Q ring, over all tiles
    bool live = true;
    for (uint32_t t = blockIdx.x; t < ntiles && live; next_tile(t)) {
      if (!has) continue;
      for (int kb = 0; kb < T.nkb && live; ++kb, ++gq) {
        const int kc = (int)(T.kbeg + (int64_t)kb * OT_KB);
        const int qs = gq & 1;
        if (!mbar_wait(&Sm.q_empty[qs], ((gq >> 1) & 1u) ^ 1u, err)) {
          live = false;
          break;
        }
        mbar_expect_tx(&Sm.q_full[qs], Q_BYTES);
        for (int p = 0; p < S; ++p) tma_load_3d(&tmQ, &Sm.q_full[qs], Sm.q[qs] + p * QS_BYTES, kc, T.prow + T.l0, p);
        for (int p = 0; p < S; ++p, ++g) {
          const int ps = g % OtCfg<S, NT>::PST;
          if (!mbar_wait(&Sm.p_empty[ps], ((g / OtCfg<S, NT>::PST) & 1u) ^ 1u, err)) {
            live = false;
            break;
          }
          mbar_expect_tx(&Sm.p_full[ps], OT_P_BYTES);
          if constexpr (TR) {
            tma_load_3d(&tmP, &Sm.p_full[ps], Sm.p[ps], (int)T.r0, kc, p);
            tma_load_3d(&tmP, &Sm.p_full[ps], Sm.p[ps] + OT_P_BYTES / 2, (int)T.r0 + 64, kc, p);
          } else {
            tma_load_3d(&tmP, &Sm.p_full[ps], Sm.p[ps], kc, T.prow + (int)T.r0, p);
          }
        }
      }
    }
    if (*(volatile int*)err) {  // gave up: no bulk copy may still be landing when the CTA exits
      tma_drain_ring(Sm.p_full, OtCfg<S, NT>::PST, (int)g);
      tma_drain_ring(Sm.q_full, 2, (int)gq);
    }
  } else if (warp == 1 && lane == 0) {
    uint32_t g = 0, gq = 0, gc = 0;  // planes of P, of Q and chunks used, over all tiles
    bool live = true;
    for (uint32_t t = blockIdx.x; t < ntiles && live; next_tile(t)) {
      if (!has) continue;
      for (int c = 0; c < T.nch && live; ++c, ++gc) {
        const uint32_t bsel = gc & 1, use = gc >> 1;
        if (use > 0 && !mbar_wait(&Sm.acc_empty[bsel], (use - 1) & 1u, err)) {
          live = false;
          break;
        }
        tc_fence_after();
        const uint32_t dbase = tmem + bsel * S * NT;
        const int kb0 = OT_KB_PER_CHUNK * c;
        const int kb_end = T.nkb < kb0 + OT_KB_PER_CHUNK ? T.nkb : kb0 + OT_KB_PER_CHUNK;
        for (int kb = kb0; kb < kb_end && live; ++kb, ++gq) {
          const uint32_t qs = gq & 1;
          if (!mbar_wait(&Sm.q_full[qs], (gq >> 1) & 1u, err)) {
            live = false;
            break;
          }
          tc_fence_after();
          const uint32_t qa = smem_u32(Sm.q[qs]);
          for (int p = 0; p < S; ++p, ++g) {
            const int ps = g % OtCfg<S, NT>::PST;
            if (!mbar_wait(&Sm.p_full[ps], (g / OtCfg<S, NT>::PST) & 1u, err)) {
              live = false;
              break;
            }
            tc_fence_after();
            // the planes Q_0 .. Q_(S-1-p) lie one after another (NT rows each), and the levels
            // p .. S-1 are consecutive NT-column blocks of the buffer: all pairs (p, q) are one
            // MMA with N = NT (S - p) whose column block q lands on level p + q
            // 16 values of K are 32 bytes of a K-major row, or 16 rows of 128 bytes of the MN-major tile
            const uint32_t pa = smem_u32(Sm.p[ps]);
            const uint64_t pd = TR ? sdesc_mn_sw128(pa, OT_P_BYTES / 2) : sdesc_sw128(pa);
            constexpr uint64_t pstep = TR ? 2048 / 16 : 2;
            const uint64_t qd = sdesc_sw128(qa);
            const uint32_t idesc = idesc_bf16(OT_M, NT * (S - p)) | (TR ? 1u << 15 : 0u);
            const uint32_t d = dbase + (uint32_t)(p * NT);
#pragma unroll
            for (int k = 0; k < OT_KB / 16; ++k) {
              // the first MMA of a chunk (p = 0) overwrites every level of the buffer
              const uint32_t acc = (kb == kb0 && p == 0 && k == 0) ? 0u : 1u;
              tc_mma_bf16(d, pd + pstep * k, qd + 2ull * k, idesc, acc);
            }
            tc_commit(&Sm.p_empty[ps]);
          }
          if (live) tc_commit(&Sm.q_empty[qs]);
        }
        if (live) tc_commit(&Sm.acc_full[bsel]);
      }
    }
    if (*(volatile int*)err) {  // gave up: wait for the MMAs issued before tensor memory is freed
      tc_commit(&Sm.mma_drain);
      mbar_drain(&Sm.mma_drain, 0u);
    }
  } else if (MODE == 4 && warp >= 4) {
    // warps 4-7 the first 16 columns of a tile, warps 8-11 the others; T before the products are done
    const int ew = warp & 3, half = (warp - 4) >> 2;
    uint32_t gc = 0;
    bool ok = true;
    for (uint32_t t = blockIdx.x; t < ntiles && ok; next_tile(t)) {
      if (!has) continue;
      const int64_t r = T.r0 + ew * 32 + lane;
      const int l0 = T.l0 + 16 * half, left = T.M - l0;
      const int er = r < rows ? EP[T.prow + r] : 0;
      const int eqv = lane < 16 && lane < left ? EQ[T.prow + l0 + lane] : 0;
      double* o = static_cast<double*>(out) + (int64_t)T.z * tri.mstride + (int64_t)l0 * ldo + r;
      double tv[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) tv[j] = r < rows && j < left && r >= l0 + j ? o[(int64_t)j * ldo] : 0.0;
      const uint32_t bsel = gc & 1, use = gc >> 1;
      ++gc;
      if (!__all_sync(0xffffffffu, mbar_wait(&Sm.acc_full[bsel], use & 1u, err))) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t base = tmem + ((uint32_t)(ew * 32) << 16) + bsel * S * NT + 16 * half;
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        uint32_t v[OZ_S][8];
#pragma unroll
        for (int q = 0; q < OZ_S; ++q) tmem_ld8_nowait(base + (uint32_t)(q * NT + 8 * g), v[q]);
        tmem_wait_ld();
        if (g == 1) {
          tc_fence_before();
          mbar_arrive(&Sm.acc_empty[bsel]);  // every sum of the thread's columns is in registers
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int j = 8 * g + q;
          int L[OZ_S];
#pragma unroll
          for (int p = 0; p < OZ_S; ++p) L[p] = __float2int_rz(__uint_as_float(v[p][q]));  // exact integers
          const long long hi = (long long)(L[0] * 128 + L[1]) * 16384 + (L[2] * 128 + L[3]);
          const long long lo = (long long)(L[4] * 128 + L[5]) * 16384 + (L[6] * 128 + L[7]);
          const int eq = __shfl_sync(0xffffffffu, eqv, j), e = er + eq;
          // the two scaled terms from the integers' bits: the float64 pipe only adds and subtracts
          bool fine = true;
          const double shi = i53_scaled(hi, e - 35, &fine), slo = i53_scaled(lo, e - 63, &fine);
          double d = shi + slo;
          if (oz_bad(er) || oz_bad(eq)) d = __longlong_as_double(0x7ff8000000000000ll);
          else if (!fine) d = ldexp(fma((double)lo, 0x1p-63, (double)hi * 0x1p-35), e);
          if (r < rows && j < left && r >= l0 + j) o[(int64_t)j * ldo] = tv[j] - d;
        }
      }
    }
  } else if (MODE != 4 && warp >= 4) {
    const int ew = warp - 4;
    uint32_t gc = 0;  // chunks read, over all tiles
    bool ok = true;
    for (uint32_t t = blockIdx.x; t < ntiles && ok; next_tile(t)) {
      if (!has) continue;
      // what the last step needs besides the sums, on its way while the products are formed
      const int64_t r = T.r0 + ew * 32 + lane;
      const bool mine = r < rows;
      const int er = mine ? EP[T.prow + r] : 0;
      const double br = MODE == 0 && mine ? b[r] : 0.0;
      int eqv[NT / 32];  // of column 32 h + lane
      double cv[NT / 32];
#pragma unroll
      for (int h = 0; h < NT / 32; ++h) {
        const int l = T.l0 + 32 * h + lane;
        eqv[h] = l < T.M ? EQ[T.prow + l] : 0;
        cv[h] = MODE == 2 && coef && l < T.M ? coef[l] : 0.0;
      }
      // S = 8 (float64-accurate): the chunk's 8 exact level sums (|L_t| <= (t+1) 2^20, so L0 128 + L1 and
      // the like fit an int) are added exactly into two int64 accumulators per column, hi += L0 2^21 +
      // L1 2^14 + L2 2^7 + L3 and lo likewise from L4 .. L7 (value = hi 2^-35 + lo 2^-63; each under 2^44 per
      // chunk, so exact for K <= 2^27 per split), 8 columns at a time -- integer work, off GB300's slow float64
      // pipe -- and turned into one double at the end.  S = 4: float32 accumulators.
      Acc acc[S == OZ_S ? 1 : NT];
      long long hacc[S == OZ_S ? NT : 1], lacc[S == OZ_S ? NT : 1];
#pragma unroll
      for (int j = 0; j < (S == OZ_S ? 1 : NT); ++j) acc[j] = Acc(0);
#pragma unroll
      for (int j = 0; j < (S == OZ_S ? NT : 1); ++j) hacc[j] = lacc[j] = 0;
      for (int c = 0; c < T.nch; ++c, ++gc) {
        const uint32_t bsel = gc & 1, use = gc >> 1;
        if (!__all_sync(0xffffffffu, mbar_wait(&Sm.acc_full[bsel], use & 1u, err))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t base = tmem + ((uint32_t)(ew * 32) << 16) + bsel * S * NT;
        if constexpr (S == OZ_S) {
#pragma unroll
          for (int g = 0; g < NT / 8; ++g) {
            uint32_t v[OZ_S][8];
#pragma unroll
            for (int t = 0; t < OZ_S; ++t) tmem_ld8_nowait(base + (uint32_t)(t * NT + 8 * g), v[t]);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              int L[OZ_S];
#pragma unroll
              for (int t = 0; t < OZ_S; ++t) L[t] = __float2int_rz(__uint_as_float(v[t][j]));  // exact integers
              hacc[8 * g + j] += (long long)(L[0] * 128 + L[1]) * 16384 + (L[2] * 128 + L[3]);
              lacc[8 * g + j] += (long long)(L[4] * 128 + L[5]) * 16384 + (L[6] * 128 + L[7]);
            }
          }
        } else {
#pragma unroll 1
          for (int t = S - 1; t >= 0; --t) {  // smallest level first
#pragma unroll
            for (int h = 0; h < NT / 32; ++h) {
              uint32_t v[32];
              tmem_ld32_nowait(base + (uint32_t)(t * NT + 32 * h), v);
              tmem_wait_ld();
              const float sc = __int_as_float((127 - 7 * (t + 2)) << 23);  // 2^(-7(t+2)), exact
#pragma unroll
              for (int j = 0; j < 32; ++j) acc[32 * h + j] = fmaf(__uint_as_float(v[j]), sc, acc[32 * h + j]);
            }
          }
        }
        tc_fence_before();
        mbar_arrive(&Sm.acc_empty[bsel]);
      }
      if (ok) {
        using TU = typename std::conditional<S == OZ_S, double, float>::type;
        // G columns at a time: U is read G ahead (one by one a load waits for the last store), and the
        // columns' float64 arithmetic overlaps
        constexpr int G = S == OZ_S ? 4 : 8;
        const double sign = MODE == 3 ? tri.sign : 1.0;
        // the tile's first value: row r of its column l0
        TU* o = nullptr;
        double* o64 = nullptr;
        if (MODE == 0) o64 = static_cast<double*>(out) + (int64_t)T.l0 * ldo + r;
        else if (MODE == 1) o64 = static_cast<double*>(out) + ((int64_t)T.z * T.M + T.l0) * ldo + r;
        else if (MODE == 2) o = static_cast<TU*>(out) + (int64_t)T.l0 * ldo + r;
        else
          o = static_cast<TU*>(out) + (int64_t)(T.z / tri.pairs) * tri.mstride +
              (int64_t)(T.z % tri.pairs) * tri.pstride + (int64_t)T.l0 * ldo + r;
#pragma unroll
        for (int j0 = 0; j0 < NT; j0 += G) {
          const int left = T.M - T.l0 - j0;  // columns from here
          if (left <= 0) break;
          TU uv[G];
          if (MODE == 2 && coef) {
#pragma unroll
            for (int q = 0; q < G; ++q) uv[q] = mine && q < left ? o[(int64_t)(j0 + q) * ldo] : TU(0);
          }
#pragma unroll
          for (int q = 0; q < G; ++q) {
            const int j = j0 + q;
            const int eq = __shfl_sync(0xffffffffu, eqv[j / 32], j % 32), e = er + eq;
            const bool bad = oz_bad(er) || oz_bad(eq);
            if constexpr (MODE == 3 && S != OZ_S) {
              // a float32 result needs no float64 arithmetic: one scaling by a power of two, rounded once
              const float sg = (float)sign * acc[j];
              const float v = bad ? __int_as_float(0x7fc00000)
                                  : (e >= -126 && e <= 127 ? sg * __int_as_float((127 + e) << 23) : ldexpf(sg, e));
              if (mine && q < left) o[(int64_t)j * ldo] = v;
            } else {
              double d;
              if constexpr (S == OZ_S) d = fma((double)lacc[j], 0x1p-63, (double)hacc[j] * 0x1p-35);
              else d = (double)acc[j];
              const double v = bad ? __longlong_as_double(0x7ff8000000000000ll)
                                   : (e >= -1022 && e <= 1023 ? d * pow2d(e) : ldexp(d, e));
              const double cf = MODE == 2 ? __shfl_sync(0xffffffffu, cv[j / 32], j % 32) : 0.0;
              if (mine && q < left) {
                if (MODE == 0) o64[(int64_t)j * ldo] = br - v;
                else if (MODE == 1) o64[(int64_t)j * ldo] = v;
                else if (MODE == 3) o[(int64_t)j * ldo] = (TU)(sign * v);
                else o[(int64_t)j * ldo] = coef ? (TU)(v + cf * (double)uv[q]) : (TU)v;
              }
            }
          }
        }
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// One CTA per slot of the GPU at most
template <int S, int NT>
unsigned ot_grid(const OtTiles& t) {
  return (unsigned)std::min<int64_t>((int64_t)t.gx * t.gy * t.gz, 152 * OtCfg<S, NT>::CTAS_PER_SM);
}

// 3D map over the slice planes (K fastest, then rows, then the plane index),
// box = 64 values of K x box_rows x 1 plane, 128-byte swizzle.  ld, plane: values from one row and one plane to the
// next where the map covers a part of larger planes (0: kp and rows kp).
tk_status make_slice_map(CUtensorMap* map, const void* base, int64_t rows, int64_t kp, uint32_t box_rows, int planes,
                         int64_t ld = 0, int64_t plane = 0) {
  if (ld == 0) ld = kp;
  if (plane == 0) plane = rows * ld;
  EncodeTiledFn fn;
  TK_TRY(encode_fn(&fn));
  const cuuint64_t dims[3] = {(cuuint64_t)kp, (cuuint64_t)rows, (cuuint64_t)planes};
  const cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)plane * 2};
  const cuuint32_t box[3] = {(cuuint32_t)OT_KB, box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error_msg("cuTensorMapEncodeTiled rejected the slice layout");
    return TK_ECUDA;
  }
  return TK_OK;
}

// P: planesP digit planes of rows x K, Q: planesQ planes of M x K (both K
// rounded up to 64); S digits of each are used.
// The lambda-tile width of a product with M rows of the small operand: 64 for the
// LSQR products (S = 4) over more than 32 lambda, else 32.
constexpr int oz_tile_n(int S, int64_t M) { return (S != OZ_S && M > 32) ? 64 : 32; }

// The big operand of a product: K-major planes of rows x K (trans = false), or MN-major: the planes
// hold K x rows (trans = true).
struct OtBig {
  const void* planes;
  const int* E;  // exponents of its `rows`
  int64_t rows, K;
  bool trans;
  int64_t ld = 0, plane = 0;  // strides of larger planes that it is a part of (as make_slice_map)
};

template <int S, int MODE, int NT, bool TR, bool SYM>
tk_status launch_oz_tc_nt(const OtBig& P, const void* Qs, const int* EQ, int M, int planesQ, int64_t kp, int64_t kps,
                          int sp, const double* b, void* out, int64_t ldo, const double* coef, int* err,
                          cudaStream_t st) {
  CUtensorMap mP, mQ;
  if (TR) TK_TRY(make_slice_map(&mP, P.planes, P.K, cdiv(P.rows, OZ_KPAD) * OZ_KPAD, OT_KB, OZ_S, P.ld, P.plane));
  else TK_TRY(make_slice_map(&mP, P.planes, P.rows, kp, OT_M, OZ_S, P.ld, P.plane));
  TK_TRY(make_slice_map(&mQ, Qs, M, kp, NT, planesQ));
  const size_t smem = sizeof(OtSmem<S, NT>) + 1024;
  TK_CUDA(cudaFuncSetAttribute(k_oz_tc<S, MODE, NT, TR, SYM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const OtTiles tl{(uint32_t)cdiv(P.rows, OT_M), (uint32_t)cdiv(M, NT), (uint32_t)sp};
  if ((double)tl.gx * tl.gy * tl.gz > 2e9) {
    set_error_msg("digit product: too many tiles for one launch");
    return TK_EINVAL;
  }
  const unsigned grid = SYM ? tl.gx * tl.gy * tl.gz : ot_grid<S, NT>(tl);
  k_oz_tc<S, MODE, NT, TR, SYM>
      <<<grid, 256, smem, st>>>(mP, mQ, P.E, EQ, P.rows, M, kp, kps, b, out, ldo, coef, err, tl, OtTri{});
  TK_LAUNCH_CHECK();
  return TK_OK;
}

template <int S, int MODE, bool TR, bool SYM = false>
tk_status launch_oz_tc(const OtBig& P, const void* Qs, const int* EQ, int M, int planesQ, int splits, const double* b,
                       void* out, int64_t ldo, const double* coef, int* err, cudaStream_t st) {
  const int64_t K = P.K, kp = cdiv(K, OZ_KPAD) * OZ_KPAD;
  if (P.rows > INT32_MAX - 2 * OT_M || kp > INT32_MAX || M > 65535 * OT_N) {
    set_error_msg("emulated product: dimensions exceed the 32-bit TMA coordinates");
    return TK_EINVAL;
  }
  const int64_t kps = cdiv(cdiv(K, splits), OT_CHUNK) * OT_CHUNK;  // whole chunks per split
  const int sp = (int)cdiv(K, kps);
  if (S == OZ_S && kps > OT_MAX_KPS) {  // the exact int64 level accumulators of a split
    set_error_msg("emulated product: more than 2^27 values of K in one split");
    return TK_EINVAL;
  }
  if (oz_tile_n(S, M) == 64) {
    if constexpr (S != OZ_S)
      TK_TRY((launch_oz_tc_nt<S, MODE, 64, TR, SYM>(P, Qs, EQ, M, planesQ, kp, kps, sp, b, out, ldo, coef, err, st)));
  } else {
    TK_TRY((launch_oz_tc_nt<S, MODE, 32, TR, SYM>(P, Qs, EQ, M, planesQ, kp, kps, sp, b, out, ldo, coef, err, st)));
  }
  if (MODE == 1 && sp < splits) {  // the caller sums `splits` planes: the unused ones are zero
    double* o = static_cast<double*>(out);
    TK_CUDA(cudaMemsetAsync(o + (int64_t)sp * M * ldo, 0, sizeof(double) * (size_t)(splits - sp) * M * ldo, st));
  }
  return TK_OK;
}

// ---- a level of the triangular inverse -----------------------------------------
// Digit planes (row stride h) and row exponents of the blocks of a level: batch z = (matrix l, pair i),
// row r: src + l mstride + i pstride + r ld, h values; rows or columns past the matrix (r or k >= n - edge,
// edge = (2 i + 1) h, where row_edge / col_edge is set) and, with lower, the columns k > r are zero.
// shift (per matrix n exponents, by the pair's diagonal index): value k counts 2^shift[k] times.
template <typename T>
__global__ void __launch_bounds__(256)
    k_oz_block_rows(const T* __restrict__ src, int64_t mstride, int64_t pstride, int64_t ld, int pairs, int h, int n,
                    int row_edge, int col_edge, int lower, const int* __restrict__ shift, int64_t rows, int planes,
                    int* __restrict__ E, __nv_bfloat16* __restrict__ out) {
  __shared__ int sh[8];
  const int z = blockIdx.y, r = blockIdx.x;
  const int left = n - (2 * (z % pairs) + 1) * h;
  const T* x = src + (int64_t)(z / pairs) * mstride + (int64_t)(z % pairs) * pstride + (int64_t)r * ld;
  int K = h;
  if (col_edge && left < K) K = left;
  if (lower && r + 1 < K) K = r + 1;
  if (row_edge && r >= left) K = 0;
  if (K < 0) K = 0;
  bool bad = false;
  if (shift) shift += (int64_t)(z / pairs) * n + 2 * (int64_t)(z % pairs) * h;
  int e = oz_vec_exp<T>(x, shift, 0, K, &bad);
  e = oz_block_exp(e, bad, sh);
  const int64_t row = (int64_t)z * h + r;
  if (threadIdx.x == 0) E[row] = e;
  unsigned* o = reinterpret_cast<unsigned*>(out + row * h);
  for (int k = 2 * threadIdx.x; k < h; k += 2 * blockDim.x)
    oz_vec_split<T>(x, shift, k, K, e, rows * h, planes, o + k / 2);
}
// up[l][k] = the exponent of R_kk, down[l][k] its negative (0 where R_kk is not a positive finite number)
__global__ void __launch_bounds__(256)
    k_oz_diag_exp(const double* __restrict__ R, int64_t ldr, int64_t rstride, int n, int* __restrict__ up,
                  int* __restrict__ down) {
  const int k = blockIdx.x * 256 + threadIdx.x, l = blockIdx.y;
  if (k >= n) return;
  const double d = R[(int64_t)l * rstride + (int64_t)k * (ldr + 1)];
  const int e = d > 0.0 && d <= 1.7976931348623157e308 ? ilogb(d) : 0;
  up[(int64_t)l * n + k] = e;
  down[(int64_t)l * n + k] = -e;
}
// M[a + r][a + h + l] = Mt[a + h + l][a + r] for the level's blocks (a = 2 i h): 32 x 32 tiles
template <typename T>
__global__ void __launch_bounds__(256)
    k_oz_block_transpose(const T* __restrict__ Mt, T* __restrict__ M, int64_t ldm, int64_t mstride, int pairs, int h,
                         int n) {
  __shared__ T tile[32][33];
  const int z = blockIdx.z, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t a = 2 * (int64_t)(z % pairs) * h;
  const int64_t l0 = a + h + (int64_t)blockIdx.y * 32, r0 = a + (int64_t)blockIdx.x * 32;
  if (l0 >= n) return;
  const T* src = Mt + (int64_t)(z / pairs) * mstride;
  T* dst = M + (int64_t)(z / pairs) * mstride;
  for (int q = ty; q < 32; q += 8) tile[q][tx] = src[(l0 + q) * ldm + r0 + tx];
  __syncthreads();
  for (int q = ty; q < 32; q += 8) dst[(r0 + q) * ldm + l0 + tx] = tile[tx][q];
}

// ---- Cholesky trailing update -------------------------------------------------
// Right-looking blocked Cholesky (upper, R^T R = C + lambda I), 64-row block
// step kb: with the row panel P = R[kb rows, columns > kb] (64 x w) already
// solved, the trailing upper triangle T -= P^T P.  The panel's columns are
// sliced with one exponent per column (the output index), stored K-major
// (planes [lambda][p][column][64]); one CTA then forms a 128 x 64 tile of
// P^T P for one lambda from all 8 + 8 slice planes at once (K = 64: a single
// chunk, exact in FP32), flushes the 8 levels into float64 and subtracts the
// scaled result from T through shared memory (coalesced).

// Panel slices of block row kb for every lambda (grid: column tiles of 32 x
// lambda).  Rows c >= w of the slice planes are not written.
__global__ void __launch_bounds__(256) k_oz_panel_slice(const double* __restrict__ R, int64_t ldr, int64_t rstride,
                                                        int64_t np, int kb, __nv_bfloat16* __restrict__ out,
                                                        int* __restrict__ EC) {
  __shared__ double tile[64][33];
  __shared__ int ex[32];
  const int l = blockIdx.y;
  const int64_t c0 = (int64_t)(kb + 1) * 64, w = np - c0;
  const int64_t ct = (int64_t)blockIdx.x * 32;
  const double* Rl = R + (int64_t)l * rstride + (int64_t)kb * 64 * ldr + c0;
  for (int idx = threadIdx.x; idx < 64 * 32; idx += blockDim.x) {
    const int k = idx >> 5, cc = idx & 31;
    const int64_t c = ct + cc;
    tile[k][cc] = c < w ? Rl[(int64_t)k * ldr + c] : 0.0;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    double mx = 0.0;
    for (int k = 0; k < 64; ++k) mx = oz_absmax(mx, tile[k][threadIdx.x]);
    const int e = oz_exponent(mx);
    ex[threadIdx.x] = e;
    const int64_t c = ct + threadIdx.x;
    if (c < w) EC[(int64_t)l * np + c] = e;
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < 64 * 32; idx += blockDim.x) {
    const int cc = idx >> 6, k = idx & 63;
    const int64_t c = ct + cc;
    if (c < w) {
      unsigned short sl[OZ_S];
      oz_split(tile[k][cc], ex[cc], sl);
      unsigned short* o = reinterpret_cast<unsigned short*>(out);
#pragma unroll
      for (int p = 0; p < OZ_S; ++p) o[(((int64_t)l * OZ_S + p) * np + c) * 64 + k] = sl[p];
    }
  }
}

// The panel's planes for the products of 256 rows: block row kb0 .. kb0 + 3, columns c from (kb0 + 4) 64 on, one
// exponent per column, planes [p][lambda np + c][256].
constexpr size_t kPanelSmem = 256 * 33 * sizeof(double);
__global__ void __launch_bounds__(256) k_oz_panel256(const double* __restrict__ R, int64_t ldr, int64_t rstride,
                                                     int64_t np, int kb0, int64_t rows, __nv_bfloat16* __restrict__ out,
                                                     int* __restrict__ EC) {
  extern __shared__ double panel[];  // [256][33]
  __shared__ double part[8][32];
  __shared__ int ex[32];
  const int l = blockIdx.y, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t c0 = (int64_t)(kb0 + 4) * 64, w = np - c0;
  const int64_t ct = (int64_t)blockIdx.x * 32;
  const double* Rl = R + (int64_t)l * rstride + (int64_t)kb0 * 64 * ldr + c0 + ct;
  double mx = 0.0;
  for (int k = ty; k < 256; k += 8) {
    const double v = ct + tx < w ? Rl[(int64_t)k * ldr + tx] : 0.0;
    panel[k * 33 + tx] = v;
    mx = oz_absmax(mx, v);
  }
  part[ty][tx] = mx;
  __syncthreads();
  if (ty == 0) {
    for (int q = 1; q < 8; ++q) mx = oz_absmax(mx, part[q][tx]);
    ex[tx] = oz_exponent(mx);
    if (ct + tx < w) EC[(int64_t)l * np + ct + tx] = ex[tx];
  }
  __syncthreads();
  unsigned* o = reinterpret_cast<unsigned*>(out);
  for (int idx = threadIdx.x; idx < 32 * 128; idx += blockDim.x) {
    const int cc = idx >> 7, k = 2 * (idx & 127);
    if (ct + cc < w) {
      unsigned short s0[OZ_S], s1[OZ_S];
      oz_split(panel[k * 33 + cc], ex[cc], s0);
      oz_split(panel[(k + 1) * 33 + cc], ex[cc], s1);
#pragma unroll
      for (int p = 0; p < OZ_S; ++p)
        o[(((int64_t)p * rows + (int64_t)l * np + ct + cc) * 256 + k) / 2] = oz_pack(s0[p], s1[p]);
    }
  }
}

constexpr int CS_M = 128;                        // rows of a CTA's slab
constexpr int CS_N = 32;                         // columns of one tile
constexpr int CS_TILES = 8;                      // column tiles per CTA
constexpr uint32_t CS_P_BYTES = CS_M * 64 * 2;   // 16 KiB per digit plane of the slab
constexpr uint32_t CS_Q_BYTES = CS_N * 64 * 2;   // 4 KiB per digit plane of a tile
constexpr uint32_t CS_TMEM_COLS = 2 * OZ_LV * CS_N;  // two buffers of 8 levels x 32 columns

struct CsSmem {
  uint8_t p[OZ_S][CS_P_BYTES];
  uint8_t q[2][OZ_S * CS_Q_BYTES];
  int ecol[CS_TILES * CS_N];  // the column exponents of the CTA's tiles
  uint64_t p_full;
  uint64_t q_full[2];
  uint64_t q_empty[2];
  uint64_t acc_full[2];
  uint64_t acc_empty[2];
  uint64_t mma_drain;  // error path: completes when every MMA the CTA issued is done
  uint32_t tmem_base;
};

// A level sum of K = 64 products (|L| <= 8 * 64 * 64 * 64 = 2^21) as an
// int: the float's integer read back through the 1.5 * 2^23 offset (exact for
// |L| < 2^22).
__device__ __forceinline__ int level_int(uint32_t bits) {
  return __float_as_int(__fadd_rn(__uint_as_float(bits), 12582912.0f)) - 0x4B400000;
}

// 32 consecutive bytes (32-byte aligned) of global memory
__device__ __forceinline__ void ld_global_v4(const double* p, double* v) {
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3])
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void st_global_v4(double* p, const double* v) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3])
               : "memory");
}

// Grid: (row slabs of 128, chunks of 8 column tiles of 32, lambda) over the
// w x w trailing block.  Slab i0 needs the tiles j0 >= i0 (j >= i); a CTA
// whose chunk holds none exits at once.  The slab's digit planes are loaded
// once; the tiles stream through a 2-slot ring and two tensor-memory buffers,
// so the flush and the update of one tile overlap the products of the next.
// Flush: the 8 exact level sums are combined in int64 by Horner,
// hi = ((L0 128 + L1) 128 + L2) 128 + L3 and lo likewise from L4..L7 (both
// below 2^43), and the tile value is hi 2^-35 + lo 2^-63 (exact products of
// exact integers), scaled by 2^(E_i + E_j).
__global__ void __launch_bounds__(384, 1)
    k_oz_syrk(const __grid_constant__ CUtensorMap tmP, const __grid_constant__ CUtensorMap tmQ,
              const int* __restrict__ EC, int64_t np, int kb, int rem, double* __restrict__ R, int64_t ldr,
              int64_t rstride, int* __restrict__ err) {
  extern __shared__ __align__(1024) uint8_t cs_raw[];
  CsSmem& S = *reinterpret_cast<CsSmem*>((reinterpret_cast<uintptr_t>(cs_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int l = blockIdx.z;
  const int64_t c0 = (int64_t)(kb + 1) * 64, w = np - c0;
  const int i0 = (int)blockIdx.x * CS_M;
  const int t_first = i0 / CS_N + (int)blockIdx.y * CS_TILES;
  const int t_all = (int)(w / CS_N);
  const int nt = t_all - t_first < CS_TILES ? t_all - t_first : CS_TILES;
  if (nt <= 0) return;

  if (threadIdx.x == 0) {
    mbar_init(&S.p_full, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(&S.q_full[s], 1);
      mbar_init(&S.q_empty[s], 1);
      mbar_init(&S.acc_full[s], 1);
      mbar_init(&S.acc_empty[s], 256);
    }
    mbar_init(&S.mma_drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem_base)),
                 "r"(CS_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem_base;

  if (warp == 0 && lane == 0) {
    mbar_expect_tx(&S.p_full, OZ_S * CS_P_BYTES);
    for (int p = 0; p < OZ_S; ++p) tma_load_3d(&tmP, &S.p_full, S.p[p], 0, i0, l * OZ_S + p);
    int gq = 0;  // tiles issued into the Q ring
    for (int t = 0; t < nt; ++t) {
      const int s = t & 1;
      if (!mbar_wait(&S.q_empty[s], ((uint32_t)(t >> 1) & 1u) ^ 1u, err)) break;
      mbar_expect_tx(&S.q_full[s], OZ_S * CS_Q_BYTES);
      const int j0 = (t_first + t) * CS_N;
      for (int p = 0; p < OZ_S; ++p) tma_load_3d(&tmQ, &S.q_full[s], S.q[s] + p * CS_Q_BYTES, 0, j0, l * OZ_S + p);
      ++gq;
    }
    if (*(volatile int*)err) {  // gave up: no bulk copy may still be landing when the CTA exits
      mbar_drain(&S.p_full, 0u);
      tma_drain_ring(S.q_full, 2, gq);
    }
  } else if (warp == 1 && lane == 0) {
    if (mbar_wait(&S.p_full, 0u, err)) {
      for (int t = 0; t < nt; ++t) {
        const int s = t & 1;
        if (!mbar_wait(&S.q_full[s], (uint32_t)(t >> 1) & 1u, err)) break;
        if (t >= 2 && !mbar_wait(&S.acc_empty[s], (uint32_t)((t >> 1) - 1) & 1u, err)) break;
        tc_fence_after();
        const uint64_t qd = sdesc_sw128(smem_u32(S.q[s]));
        const uint32_t dbase = tmem + (uint32_t)(s * OZ_LV * CS_N);
        for (int p = 0; p < OZ_S; ++p) {
          // planes Q_0 .. Q_(7-p) are contiguous: one MMA of N = 32 (8 - p) onto levels p .. 7
          const uint64_t pd = sdesc_sw128(smem_u32(S.p[p]));
          const uint32_t idesc = idesc_bf16(CS_M, CS_N * (OZ_S - p));
          const uint32_t d = dbase + (uint32_t)(p * CS_N);
#pragma unroll
          for (int k = 0; k < 4; ++k) tc_mma_bf16(d, pd + 2ull * k, qd + 2ull * k, idesc, (p == 0 && k == 0) ? 0u : 1u);
        }
        tc_commit(&S.q_empty[s]);
        tc_commit(&S.acc_full[s]);
      }
    }
    if (*(volatile int*)err) {  // gave up: wait for the MMAs issued before tensor memory is freed
      tc_commit(&S.mma_drain);
      mbar_drain(&S.mma_drain, 0u);
    }
  } else if (warp >= 4) {
    // 8 epilogue warps: warp w reads tensor-memory lanes 32 (w % 4) .. (the rows), and the two warps
    // of a lane quarter split each tile's 32 columns: warps 4-7 the first 16, warps 8-11 the last 16
    const int ew = warp & 3, half = (warp - 4) >> 2;
    const int64_t i = i0 + ew * 32 + lane;
    const bool mine = i < rem;  // (rem <= w)
    const int* El = EC + (int64_t)l * np;
    const int ei = mine ? El[i] : 0;
    double* Trow = R + (int64_t)l * rstride + (c0 + i) * ldr + c0;
    // the exponents of the CTA's columns, once, in shared memory (the epilogue warps only)
    for (int c = (int)threadIdx.x - 128; c < CS_TILES * CS_N; c += 256) {
      const int64_t col = (int64_t)t_first * CS_N + c;
      S.ecol[c] = col < w ? El[col] : 0;
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    // the thread's 16 columns of a tile in 2 groups of 8; per group the 8 levels of the 8 columns are
    // read from tensor memory and the exact integers hi = L0 2^21 + L1 2^14 + L2 2^7 + L3 and lo (L4 ..
    // L7 likewise) formed as (L0 128 + L1) 2^14 + (L2 128 + L3) -- the same integers as a Horner
    // chain, |L0 128 + L1| < 2^30
    constexpr int G = 8;
    for (int t = 0; t < nt; ++t) {
      const int s = t & 1;
      const int64_t j0 = (int64_t)(t_first + t) * CS_N + half * 2 * G;
      // a thread's 16 columns are 128 consecutive bytes of its row of T: four 32-byte loads and stores (whole
      // sectors; element by element every 8-byte store was a partial sector write of its own: order 4096, 64
      // lambda 2.51 ms a step on average, now 2.10; order 2048, 32 lambda 0.36, now 0.30).  Tiles on
      // the diagonal (columns below the thread's row) and marked rows go element by element.
      const bool full = mine && j0 >= i;
      // T of the thread's 16 columns first: their loads do not wait for the products
      double tv[2][G];
      if (full) {
#pragma unroll
        for (int q = 0; q < 4; ++q) ld_global_v4(Trow + j0 + 4 * q, tv[q >> 1] + 4 * (q & 1));
      } else {
#pragma unroll
        for (int gi = 0; gi < 2; ++gi)
#pragma unroll
          for (int j = 0; j < G; ++j) {
            const int64_t col = j0 + gi * G + j;
            tv[gi][j] = (mine && col < w && col >= i) ? Trow[col] : 0.0;
          }
      }
      if (!mbar_wait(&S.acc_full[s], (uint32_t)(t >> 1) & 1u, err)) break;
      tc_fence_after();
      const uint32_t base =
          tmem + ((uint32_t)(ew * 32) << 16) + (uint32_t)(s * OZ_LV * CS_N) + (uint32_t)(half * 2 * G);
#pragma unroll
      for (int gi = 0; gi < 2; ++gi) {
        const int64_t jg = j0 + gi * G;
        uint32_t v[OZ_LV][G];
#pragma unroll
        for (int lv = 0; lv < OZ_LV; ++lv) tmem_ld8_nowait(base + (uint32_t)(lv * CS_N + gi * G), v[lv]);
        tmem_wait_ld();
        if (gi == 1) {
          tc_fence_before();
          mbar_arrive(&S.acc_empty[s]);  // every level of the thread's columns is in registers
        }
        if (mine) {
#pragma unroll
          for (int j = 0; j < G; ++j) {
            const int ej = S.ecol[t * CS_N + half * 2 * G + gi * G + j];
            const int e = ei + ej;
            const int a0 = level_int(v[0][j]) * 128 + level_int(v[1][j]);
            const int a1 = level_int(v[2][j]) * 128 + level_int(v[3][j]);
            const int b0 = level_int(v[4][j]) * 128 + level_int(v[5][j]);
            const int b1 = level_int(v[6][j]) * 128 + level_int(v[7][j]);
            const long long hi = (long long)a0 * 16384 + a1, lo = (long long)b0 * 16384 + b1;
            // (hi 2^-35 + lo 2^-63) 2^e with the two scaled terms built exactly from the integers'
            // bits; the sum and the subtraction are the only float64 operations (the same rounding
            // as scaling the rounded sum, since a power of two scales exactly)
            bool ok = true;
            const double shi = i53_scaled(hi, e - 35, &ok), slo = i53_scaled(lo, e - 63, &ok);
            double r;
            if (oz_bad(ei) || oz_bad(ej)) {  // a row or column marked non-finite: NaN (its digits are zero)
              r = __longlong_as_double(0x7ff8000000000000ll);
            } else if (ok) {
              r = tv[gi][j] - (shi + slo);
            } else {  // a scaled term outside the normal range: through the float64 pipe
              const double vhi = (double)hi * 0x1p-35, vlo = (double)lo * 0x1p-63;  // exact
              r = tv[gi][j] - (vhi + vlo) * (e >= -1022 && e <= 1023 ? pow2d(e) : ldexp(1.0, e));
            }
            tv[gi][j] = r;
            if (!full && jg + j < w && jg + j >= i) Trow[jg + j] = r;
          }
          if (full) {
#pragma unroll
            for (int q = 0; q < 2; ++q) st_global_v4(Trow + jg + 4 * q, tv[gi] + 4 * q);
          }
        }
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(CS_TMEM_COLS) : "memory");
  }
}


// ---- the two products of an LSQR step, fused over one read of A -----------------
// One LSQR step of the mixed form needs U' = W A^T + c .* U (m values per lambda)
// and then G = U' A (n values per lambda).  The second product of a band of rows
// needs the first product over the band's whole rows, so a band must be held
// between the two.  Here a cluster of CL CTAs (CL a power of two <= 8) owns one
// band of 128 rows at a time, CTA q the columns [q cpc, (q + 1) cpc) of it (cpc <=
// 256, so the CTA's slab of the 4 digit planes is at most 256 KiB):
//   P1  the CTA's part of W A^T for the band (K = its columns) on tcgen05 into one
//       of two tensor-memory buffers; W's digits stay in shared memory throughout;
//   X1  the CL partials are added through distributed shared memory: CTA q adds
//       the rows [q 128/CL, (q + 1) 128/CL) in rank order, forms U' = v + c U for
//       them (written to U), and stores u' = U' 2^(E_r - E_max) (the row scale of
//       A's digits moved onto U') into every CTA's copy of the band's u';
//   X2  every CTA digitizes the band's u' (4 digits, one exponent per lambda) into
//       the B operand of
//   P2  G_q += A_slab^T u' on tcgen05, the A operand read MN-major from the same
//       digit planes, read again (from L2: a few microseconds after P1's read).
// The producer issues the next band's P1 loads before this band's P2 loads, so A
// streams from memory while the epilogue exchanges and digitizes.  Each CTA keeps
// its columns' G in registers across all the bands its cluster processes, and
// writes one partial plane per cluster at the end.  The exchange uses mbarriers in
// distributed shared memory with bounded waits; every CTA reaches the cluster
// barrier before exit, so no CTA leaves while another may still read or write its
// shared memory.
constexpr int FU_M = 128;   // band rows
constexpr int FU_NT = 32;   // lambda
constexpr int FU_RS = 3;    // ring slots of one 128-column chunk of one digit plane (2 TMA boxes)
constexpr int FU_S = 4;     // digits (the float32 LSQR products)
constexpr uint32_t FU_SLOT = 2 * OT_P_BYTES;                 // 32 KiB
constexpr uint32_t FU_QBOX = FU_NT * 64 * 2;                 // 4 KiB: 32 rows x 64 values of one plane
constexpr uint32_t FU_QCH = 2 * FU_S * FU_QBOX;              // 32 KiB: 128 K x 4 planes
constexpr uint32_t FU_TMEM_COLS = 512;                       // P1: 2 x 128, P2: 2 x 128

struct FuSmem {
  uint8_t ring[FU_RS][FU_SLOT];
  uint8_t wq[2][FU_QCH];      // W digits of chunk c (resident): [64-K box][plane][32 rows][128 B]
  uint8_t q2[FU_QCH];         // u' digits: [64-row chunk][plane][32 lambda][128 B]
  float pbuf[FU_NT * FU_M];   // P1 partial, [lambda][row]
  float ub[FU_NT * FU_M];     // u' of the band, [lambda][row]
  uint32_t umax[4][FU_NT];    // per warp: max |u'| bits per lambda
  int ea[FU_M];
  int eu[FU_NT];
  int ew[FU_NT];
  float psc[FU_NT];           // 2^(E_max + E_u) of the band, per lambda (the P2 scale)
  int emax4[4];
  uint64_t ring_full[FU_RS], ring_empty[FU_RS], w_full;
  uint64_t p1_full[2], p1_empty[2], q2_full, q2_empty, p2_full[2], p2_empty[2];
  uint64_t pb_full, pb_empty, ub_full, ub_empty;
  uint64_t mma_drain;
  uint32_t tmem_base;
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_id_x() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t nclusters_x() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
  return r;
}
// shared::cluster address of `p` (a shared variable of this CTA) in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t dsmem_addr(const void* p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void dsmem_arrive(uint32_t bar_cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster_addr) : "memory");
}
// generic pointer to `p` (a shared array of this CTA) in CTA `rank` of the cluster: plain loads and
// stores through it, which the compiler may batch (ordered after the acquiring waits, which clobber memory)
template <typename T>
__device__ __forceinline__ T* peer_ptr(T* p, uint32_t rank) {
  return static_cast<T*>(__cluster_map_shared_rank(static_cast<void*>(p), rank));
}
// bounded wait with cluster-scope acquire (data written by other CTAs before their arrive is visible)
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* b, uint32_t parity, int* err) {
  uint64_t t0 = 0;
  for (uint32_t i = 0; i < (1u << 26); ++i) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(b)), "r"(parity)
        : "memory");
    if (ok) return true;
    if (i >= 256) __nanosleep(32);
    if ((i & 255u) == 255u) {
      if (*(volatile int*)err) return false;
      const uint64_t t = global_ns();
      if (t0 == 0) t0 = t;
      else if (t - t0 > kWaitBudgetNs) break;
    }
  }
  atomicExch(err, 1);
  return false;
}
// true on every one of the 128 epilogue threads iff v is true on all of them (named barrier 1): the
// epilogue takes every exit together, so no thread is left waiting at a named barrier
__device__ __forceinline__ bool epi_all(bool v) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.and.pred q, 1, 128, p;\n selp.u32 %0, 1, 0, q;\n}"
      : "=r"(r)
      : "r"((uint32_t)v)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// K-major operand, 128-byte swizzle: byte offset of element (row, k) in a box of 64 values per row
__device__ __forceinline__ uint32_t sw128_off(int row, int k) {
  return (uint32_t)(row * 128 + ((((k >> 3) ^ (row & 7)) & 7) << 4) + ((k & 7) << 1));
}
// 2^e as a float (0 below the normal range, inf above)
__device__ __forceinline__ float pow2f(int e) {
  return e < -126 ? 0.f : (e > 127 ? __int_as_float(0x7f800000) : __int_as_float((127 + e) << 23));
}

// The 4 balanced base-128 digits of x 2^-E rounded to 28 bits (|x| < 2^E): the value
// v = round(x 2^(28 - E)) (exact scaling in float64, one rounding) written as
// d0 2^21 + d1 2^14 + d2 2^7 + d3 with d1..d3 in [-64, 63].
__device__ __forceinline__ void oz_split4(float x, int E, unsigned short (&bits)[4]) {
  int v = (int)__double2ll_rn((double)x * pow2d(28 - E));
#pragma unroll
  for (int p = 3; p >= 1; --p) {
    const int d = ((v + 64) & 127) - 64;
    bits[p] = oz_bf16_bits(d);
    v = (v - d) >> 7;
  }
  bits[0] = oz_bf16_bits(v);
}

__global__ void __launch_bounds__(256, 1)
    k_oz_fused(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW,
               const int* __restrict__ EA, const int* __restrict__ EC, const int* __restrict__ EW, int64_t m,
               int64_t n, int count, int cpc, float* __restrict__ U, int64_t ldu, const double* __restrict__ coef, double* __restrict__ partial,
               int* __restrict__ err) {
  extern __shared__ __align__(1024) uint8_t fu_raw[];
  FuSmem& S = *reinterpret_cast<FuSmem*>((reinterpret_cast<uintptr_t>(fu_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t q = cluster_rank();
  int cl_size;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(cl_size));
  const int64_t bands = (m + FU_M - 1) / FU_M;
  const int64_t zc = cluster_id_x(), ncl = nclusters_x();
  const int nb = zc < bands ? (int)((bands - 1 - zc) / ncl + 1) : 0;  // bands of this cluster
  const int nch = cpc / 128;       // 128-column chunks of this CTA (1 or 2)
  const int col0 = (int)q * cpc;   // this CTA's first column
  const int row_lo = (int)q * (FU_M / cl_size), nrows = FU_M / cl_size;  // this CTA's rows in X1

  if (threadIdx.x == 0) {
    for (int s = 0; s < FU_RS; ++s) {
      mbar_init(&S.ring_full[s], 1);
      mbar_init(&S.ring_empty[s], 1);
    }
    mbar_init(&S.w_full, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(&S.p1_full[s], 1);
      mbar_init(&S.p1_empty[s], 128);
      mbar_init(&S.p2_full[s], 1);
      mbar_init(&S.p2_empty[s], 128);
    }
    mbar_init(&S.q2_full, 1);
    mbar_init(&S.q2_empty, 1);
    mbar_init(&S.pb_full, cl_size);
    mbar_init(&S.pb_empty, cl_size);
    mbar_init(&S.ub_full, cl_size);
    mbar_init(&S.ub_empty, cl_size);
    mbar_init(&S.mma_drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x < FU_NT) S.ew[threadIdx.x] = threadIdx.x < count ? EW[threadIdx.x] : 0;
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem_base)),
                 "r"(FU_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  cluster_sync_all();  // every CTA's barriers are initialized before any remote arrive
  tc_fence_after();
  const uint32_t tmem = S.tmem_base;

  if (warp == 0 && lane == 0) {
    // ---- TMA producer: W once; then P1(band 0), and per band i: P1(band i + 1), P2(band i) -- the
    // same 4 planes x nch chunks of A each time
    int g = 0;
    mbar_expect_tx(&S.w_full, (uint32_t)nch * FU_QCH);
    for (int c = 0; c < nch; ++c)
      for (int kb = 0; kb < 2; ++kb)
        for (int p = 0; p < FU_S; ++p)
          tma_load_3d(&tmW, &S.w_full, S.wq[c] + (kb * FU_S + p) * FU_QBOX, col0 + 128 * c + 64 * kb, 0, p);
    auto load_band = [&](int j) -> bool {
      const int r0 = (int)((zc + (int64_t)j * ncl) * FU_M);
      for (int c = 0; c < nch; ++c) {
        const int k0 = col0 + 128 * c;
        for (int p = 0; p < FU_S; ++p, ++g) {
          const int s = g % FU_RS;
          if (!mbar_wait(&S.ring_empty[s], ((uint32_t)(g / FU_RS) & 1u) ^ 1u, err)) return false;
          mbar_expect_tx(&S.ring_full[s], FU_SLOT);
          tma_load_3d(&tmA, &S.ring_full[s], S.ring[s], k0, r0, p);
          tma_load_3d(&tmA, &S.ring_full[s], S.ring[s] + OT_P_BYTES, k0 + 64, r0, p);
        }
      }
      return true;
    };
    bool live = nb == 0 || load_band(0);
    for (int i = 0; i < nb && live; ++i) {
      if (i + 1 < nb) live = load_band(i + 1);
      if (live) live = load_band(i);
    }
    if (*(volatile int*)err) {
      tma_drain_ring(S.ring_full, FU_RS, g);
      mbar_drain(&S.w_full, 0u);
    }
  } else if (warp == 1 && lane == 0) {
    // ---- MMA issuer
    int g = 0, T = 0;
    bool live = mbar_wait(&S.w_full, 0u, err);
    tc_fence_after();
    // P1 of the cluster's j-th band into tensor-memory buffer j & 1
    auto p1 = [&](int j) -> bool {
      const int buf = j & 1;
      if (j >= 2 && !mbar_wait(&S.p1_empty[buf], (uint32_t)(((j - 2) >> 1) & 1), err)) return false;
      tc_fence_after();
      for (int c = 0; c < nch; ++c) {
        for (int p = 0; p < FU_S; ++p, ++g) {
          const int s = g % FU_RS;
          if (!mbar_wait(&S.ring_full[s], (uint32_t)(g / FU_RS) & 1u, err)) return false;
          tc_fence_after();
          const uint32_t idesc = idesc_bf16(FU_M, FU_NT * (FU_S - p));
#pragma unroll
          for (int ks = 0; ks < 8; ++ks) {  // K = 128 columns: 4 steps in each 64-column box
            const uint32_t box = (uint32_t)(ks >> 2), kk = (uint32_t)(ks & 3);
            const uint64_t ad = sdesc_sw128(smem_u32(S.ring[s]) + box * OT_P_BYTES) + 2ull * kk;
            const uint64_t bd = sdesc_sw128(smem_u32(S.wq[c]) + box * FU_S * FU_QBOX) + 2ull * kk;
            const uint32_t acc = (c == 0 && p == 0 && ks == 0) ? 0u : 1u;
            tc_mma_bf16(tmem + 128u * (uint32_t)buf + (uint32_t)(p * FU_NT), ad, bd, idesc, acc);
          }
          tc_commit(&S.ring_empty[s]);
        }
      }
      tc_commit(&S.p1_full[buf]);
      return true;
    };
    if (live && nb > 0) live = p1(0);
    for (int i = 0; i < nb && live; ++i) {
      if (i + 1 < nb && !p1(i + 1)) break;
      // P2: wait for the band's u' digits
      if (!mbar_wait(&S.q2_full, (uint32_t)(i & 1), err)) break;
      tc_fence_after();
      for (int c = 0; c < nch && live; ++c, ++T) {
        const int bsel = T & 1, use = T >> 1;
        if (use > 0 && !mbar_wait(&S.p2_empty[bsel], (uint32_t)((use - 1) & 1), err)) {
          live = false;
          break;
        }
        tc_fence_after();
        const uint32_t dbase = tmem + 256u + 128u * (uint32_t)bsel;
        for (int p = 0; p < FU_S; ++p, ++g) {
          const int s = g % FU_RS;
          if (!mbar_wait(&S.ring_full[s], (uint32_t)(g / FU_RS) & 1u, err)) {
            live = false;
            break;
          }
          tc_fence_after();
          // A operand = the slab's columns (M) x the band's rows (K), MN-major; transpose bit 15
          const uint32_t idesc = idesc_bf16(FU_M, FU_NT * (FU_S - p)) | (1u << 15);
#pragma unroll
          for (int ks = 0; ks < 8; ++ks) {  // K = 128 band rows: 16 rows (2 KiB) per step
            const uint64_t ad = sdesc_mn_sw128(smem_u32(S.ring[s]) + (uint32_t)ks * 2048u, OT_P_BYTES);
            const uint64_t bd =
                sdesc_sw128(smem_u32(S.q2) + (uint32_t)(ks >> 2) * FU_S * FU_QBOX) + 2ull * (uint32_t)(ks & 3);
            tc_mma_bf16(dbase + (uint32_t)(p * FU_NT), ad, bd, idesc, (p == 0 && ks == 0) ? 0u : 1u);
          }
          tc_commit(&S.ring_empty[s]);
        }
        if (live) tc_commit(&S.p2_full[bsel]);
      }
      if (live) tc_commit(&S.q2_empty);  // the band's u' digits are no longer read
    }
    if (*(volatile int*)err) {
      tc_commit(&S.mma_drain);
      mbar_drain(&S.mma_drain, 0u);
    }
  } else if (warp >= 4) {
    // ---- epilogue warps (thread e = TMEM lane e: a band row in P1, X2; a column in P2)
    const int e = (int)threadIdx.x - 128, ew = warp - 4;
    float gacc[2][FU_NT];
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int l = 0; l < FU_NT; ++l) gacc[c][l] = 0.f;
    bool ok = true;
    int T = 0;
    // P2 of the previous band: G of this CTA's columns += A_slab^T u', the levels weighted by
    // 2^(-7 (t + 2)), the sum by 2^(E_max + E_u) (S.psc, still the previous band's)
    auto p2_read = [&]() -> bool {
#pragma unroll
      for (int c = 0; c < 2; ++c) {  // nch <= 2, unrolled so that gacc stays in registers
        if (c >= nch) break;
        const int bsel = T & 1, use = T >> 1;
        ++T;
        if (!epi_all(mbar_wait(&S.p2_full[bsel], (uint32_t)(use & 1), err))) return false;
        tc_fence_after();
        const uint32_t base = tmem + ((uint32_t)(ew * 32) << 16) + 256u + 128u * (uint32_t)bsel;
        float lev[FU_NT];
#pragma unroll
        for (int l = 0; l < FU_NT; ++l) lev[l] = 0.f;
#pragma unroll 1
        for (int t = FU_S - 1; t >= 0; --t) {
          uint32_t v[32];
          tmem_ld32_nowait(base + (uint32_t)(t * FU_NT), v);
          tmem_wait_ld();
          const float lw = __int_as_float((127 - 7 * (t + 2)) << 23);  // the level weight 2^(-7 (t + 2))
#pragma unroll
          for (int l = 0; l < FU_NT; ++l) lev[l] = fmaf(__uint_as_float(v[l]), lw, lev[l]);
        }
        tc_fence_before();
        mbar_arrive(&S.p2_empty[bsel]);
#pragma unroll
        for (int l = 0; l < FU_NT; ++l) gacc[c][l] = fmaf(lev[l], S.psc[l], gacc[c][l]);
      }
      return true;
    };
    int ea_next = nb > 0 && zc * FU_M + e < m ? EA[zc * FU_M + e] : 0;
    for (int i = 0; i < nb && ok; ++i) {
      const int64_t r0 = (zc + (int64_t)i * ncl) * FU_M;
      // the band's row exponents and their maximum over the finite rows (the next band's loaded ahead)
      const int ea_e = ea_next;
      {
        const int64_t rn = r0 + ncl * FU_M + e;
        ea_next = i + 1 < nb && rn < m ? EA[rn] : 0;
      }
      S.ea[e] = ea_e;
      const int wm = __reduce_max_sync(0xffffffffu, (r0 + e < m && !oz_bad(ea_e)) ? ea_e : INT_MIN);
      if (lane == 0) S.emax4[ew] = wm;
      epi_sync();
      int eamax = max(max(S.emax4[0], S.emax4[1]), max(S.emax4[2], S.emax4[3]));
      if (eamax == INT_MIN) eamax = 0;
      // P1 partial of this CTA's columns, row e of the band
      const int buf = i & 1;
      if (!epi_all(mbar_wait(&S.p1_full[buf], (uint32_t)((i >> 1) & 1), err))) {
        ok = false;
        break;
      }
      tc_fence_after();
      float acc[FU_NT];
#pragma unroll
      for (int l = 0; l < FU_NT; ++l) acc[l] = 0.f;
      const uint32_t lb = tmem + ((uint32_t)(ew * 32) << 16) + 128u * (uint32_t)buf;
#pragma unroll 1
      for (int t = FU_S - 1; t >= 0; --t) {
        uint32_t v[32];
        tmem_ld32_nowait(lb + (uint32_t)(t * FU_NT), v);
        tmem_wait_ld();
        const float sc = __int_as_float((127 - 7 * (t + 2)) << 23);
#pragma unroll
        for (int l = 0; l < FU_NT; ++l) acc[l] = fmaf(__uint_as_float(v[l]), sc, acc[l]);
      }
      tc_fence_before();
      mbar_arrive(&S.p1_empty[buf]);
      // my partial may be overwritten once every CTA has read the previous band's
      if (!epi_all(i == 0 || mbar_wait_cluster(&S.pb_empty, (uint32_t)((i - 1) & 1), err))) {
        ok = false;
        break;
      }
#pragma unroll
      for (int l = 0; l < FU_NT; ++l) S.pbuf[l * FU_M + e] = acc[l];
      epi_sync();
      if (e == 0) {
        asm volatile("fence.acq_rel.cluster;" ::: "memory");
        for (int r = 0; r < cl_size; ++r) dsmem_arrive(dsmem_addr(&S.pb_full, (uint32_t)r));
      }
      // the previous band's P2 while the peers' partials arrive
      if (i > 0 && !p2_read()) {
        ok = false;
        break;
      }
      // X1: my rows of the band (4 at a time), summed over the cluster in rank order; U' = v + c U;
      // u' into every CTA
      if (!epi_all(mbar_wait_cluster(&S.pb_full, (uint32_t)(i & 1), err) &&
                   (i == 0 || mbar_wait_cluster(&S.ub_empty, (uint32_t)((i - 1) & 1), err)))) {
        ok = false;
        break;
      }
      const int nq = nrows / 4;
      for (int v = e; v < FU_NT * nq; v += 128) {
        const int l = v / nq, row = row_lo + 4 * (v % nq);
        float4 s4 = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int r = 0; r < cl_size; ++r) {
          const float4 t4 = *reinterpret_cast<const float4*>(peer_ptr(S.pbuf, (uint32_t)r) + l * FU_M + row);
          s4.x += t4.x;
          s4.y += t4.y;
          s4.z += t4.z;
          s4.w += t4.w;
        }
        const float sv[4] = {s4.x, s4.y, s4.z, s4.w};
        float up[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int64_t grow = r0 + row + k;
          up[k] = 0.f;
          if (grow < m && l < count) {
            const int er = S.ea[row + k], eq = S.ew[l];
            const int es = er + eq;
            const double val = (oz_bad(er) || oz_bad(eq)) ? __longlong_as_double(0x7ff8000000000000ll)
                               : (es >= -1022 && es <= 1023) ? (double)sv[k] * pow2d(es)
                                                             : ldexp((double)sv[k], es);
            float* u = U + (int64_t)l * ldu + grow;
            const float un = coef ? (float)(val + coef[l] * (double)*u) : (float)val;
            *u = un;
            up[k] = oz_bad(er) ? un : un * pow2f(er - eamax);
          }
        }
        const float4 u4 = make_float4(up[0], up[1], up[2], up[3]);
        for (int r = 0; r < cl_size; ++r)
          *reinterpret_cast<float4*>(peer_ptr(S.ub, (uint32_t)r) + l * FU_M + row) = u4;
      }
      epi_sync();
      if (e == 0) {
        asm volatile("fence.acq_rel.cluster;" ::: "memory");
        for (int r = 0; r < cl_size; ++r) {
          dsmem_arrive(dsmem_addr(&S.pb_empty, (uint32_t)r));
          dsmem_arrive(dsmem_addr(&S.ub_full, (uint32_t)r));
        }
      }
      // X2: the band's u' digits (4, one exponent per lambda) into the B operand of P2; thread e = row
      if (!epi_all(mbar_wait_cluster(&S.ub_full, (uint32_t)(i & 1), err) &&
                   (i == 0 || mbar_wait(&S.q2_empty, (uint32_t)((i - 1) & 1), err)))) {
        ok = false;
        break;
      }
#pragma unroll 4
      for (int l = 0; l < FU_NT; ++l) {
        const uint32_t b = __float_as_uint(fabsf(S.ub[l * FU_M + e]));  // non-finite: >= 0x7f800000
        const uint32_t mx = __reduce_max_sync(0xffffffffu, b);
        if (lane == 0) S.umax[ew][l] = mx;
      }
      epi_sync();
      if (e < FU_NT) {
        const uint32_t mx = max(max(S.umax[0][e], S.umax[1][e]), max(S.umax[2][e], S.umax[3][e]));
        const int eu = mx >= 0x7f800000u ? OZ_EBAD : oz_exponent((double)__uint_as_float(mx));
        S.eu[e] = eu;
        S.psc[e] = oz_bad(eu) ? __int_as_float(0x7fc00000) : pow2f(eamax + eu);
      }
      epi_sync();
      {
        uint8_t* base = S.q2 + (e >> 6) * FU_S * FU_QBOX;
#pragma unroll 4
        for (int l = 0; l < FU_NT; ++l) {
          const int eu = S.eu[l];
          unsigned short bits[FU_S];
          oz_split4(oz_bad(eu) ? 0.f : S.ub[l * FU_M + e], oz_bad(eu) ? 0 : eu, bits);
#pragma unroll
          for (int p = 0; p < FU_S; ++p)
            *reinterpret_cast<unsigned short*>(base + p * FU_QBOX + sw128_off(l, e & 63)) = bits[p];
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic writes -> tensor core reads
      epi_sync();
      if (e == 0) {
        mbar_arrive(&S.q2_full);
        asm volatile("fence.acq_rel.cluster;" ::: "memory");
        for (int r = 0; r < cl_size; ++r) dsmem_arrive(dsmem_addr(&S.ub_empty, (uint32_t)r));
      }
    }
    // the last band's P2
    if (ok && nb > 0) ok = p2_read();
    // this cluster's partial plane of G: partial[z][l][col]
    if (ok) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        if (c >= nch) break;
        const int64_t col = col0 + 128 * c + e;
        if (col < n) {
          const int ec = EC[col];  // the column's scale in the digits of A
#pragma unroll
          for (int l = 0; l < FU_NT; ++l)
            if (l < count)
              partial[((int64_t)zc * count + l) * n + col] =
                  oz_bad(ec) ? __longlong_as_double(0x7ff8000000000000ll) : ldexp((double)gacc[c][l], ec);
        }
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync_all();  // no CTA leaves while a peer may still use its shared memory
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(FU_TMEM_COLS) : "memory");
  }
}

}  // namespace

size_t oz_slices_bytes(int64_t rows, int64_t cols, int planes) {
  return sizeof(__nv_bfloat16) * (size_t)planes * (size_t)rows * (size_t)(cdiv(cols, OZ_KPAD) * OZ_KPAD);
}

tk_status oz_split_vectors(const void* V, tk_dtype dt, int64_t M, int64_t K, int64_t ld, const int* shift,
                           void* slices, int* E, cudaStream_t st, int planes) {
  if (M == 0 || K == 0) return TK_OK;
  const int64_t kp = cdiv(K, OZ_KPAD) * OZ_KPAD;
  const bool f64 = dt == TK_F64;
  __nv_bfloat16* out = static_cast<__nv_bfloat16*>(slices);
  if (M > 65535) {
    set_error_msg("emulated float64 product: too many rows of the small operand");
    return TK_EINVAL;
  }
  if (K < OZ_VEC_LONG) {
    if (f64) k_oz_vec<double><<<(unsigned)M, 512, 0, st>>>((const double*)V, M, K, ld, shift, E, kp, planes, out);
    else k_oz_vec<float><<<(unsigned)M, 512, 0, st>>>((const float*)V, M, K, ld, shift, E, kp, planes, out);
    TK_LAUNCH_CHECK();
    return TK_OK;
  }
  // blocks of 2048 values or more, about 8 blocks per SM in all
  const int64_t per = std::max<int64_t>(2048, cdiv(cdiv(K * M, 8 * 152), 256) * 256);
  TK_CUDA(cudaMemsetAsync(E, 0x80, sizeof(int) * (size_t)M, st));  // OZ_EZERO
  const dim3 g((unsigned)cdiv(K, per), (unsigned)M), gs((unsigned)cdiv(kp, 512), (unsigned)M);
  if (f64) k_oz_vec_exp<double><<<g, 256, 0, st>>>((const double*)V, K, ld, shift, per, E);
  else k_oz_vec_exp<float><<<g, 256, 0, st>>>((const float*)V, K, ld, shift, per, E);
  TK_LAUNCH_CHECK();
  if (f64) k_oz_vec_slice<double><<<gs, 256, 0, st>>>((const double*)V, M, K, ld, shift, E, kp, planes, out);
  else k_oz_vec_slice<float><<<gs, 256, 0, st>>>((const float*)V, M, K, ld, shift, E, kp, planes, out);
  TK_LAUNCH_CHECK();
  return TK_OK;
}

size_t oz_colmax_bytes(int64_t cols) { return sizeof(unsigned long long) * (size_t)std::max<int64_t>(cols, 1); }

// Column exponents EC of X (and, with copy, its float32 copy): one pass over X.
static tk_status oz_column_exponents(const void* X, tk_dtype dt, int64_t rows, int64_t cols, int64_t ld, int* EC,
                                     void* colmax, float* copy, cudaStream_t st) {
  unsigned long long* mx = static_cast<unsigned long long*>(colmax);
  TK_CUDA(cudaMemsetAsync(mx, 0, sizeof(unsigned long long) * (size_t)cols, st));
  // about 8 CTAs of 256 columns per SM, each over a band of rows
  const int64_t cb = cdiv(cols, 256);
  const int64_t bands = std::max<int64_t>(1, std::min<int64_t>({cdiv(8 * 152, cb), cdiv(rows, 32), 65535}));
  const int64_t rows_per = cdiv(rows, bands);
  const dim3 gm((unsigned)cb, (unsigned)cdiv(rows, rows_per));
  if (dt == TK_F64) k_oz_colmax<double><<<gm, 256, 0, st>>>((const double*)X, rows, cols, ld, rows_per, mx, copy);
  else k_oz_colmax<float><<<gm, 256, 0, st>>>((const float*)X, rows, cols, ld, rows_per, mx, copy);
  TK_LAUNCH_CHECK();
  k_oz_colexp<<<(unsigned)cb, 256, 0, st>>>(mx, cols, EC);
  TK_LAUNCH_CHECK();
  return TK_OK;
}

tk_status oz_split_matrix(const void* A, tk_dtype dt, int64_t rows, int64_t cols, int64_t ld, void* slices, int* ER,
                          int* EC, void* colmax, float* copy, cudaStream_t st) {
  if (rows == 0 || cols == 0) return TK_OK;
  TK_TRY(oz_column_exponents(A, dt, rows, cols, ld, EC, colmax, copy, st));
  const int64_t cp = cdiv(cols, OZ_KPAD) * OZ_KPAD;
  const size_t es = dt == TK_F64 ? 8 : 4;
  // about 5 blocks per SM are resident: keep their bands within half of the 129 MB L2
  int RB = 8;
  while (RB > 1 && (size_t)RB * cols * es * 5 * 152 > (size_t)64 << 20) RB /= 2;
  const int64_t nb = cdiv(rows, RB);
  if (nb > INT32_MAX) {
    set_error_msg("emulated float64 product: too many rows for the slicing grid");
    return TK_EINVAL;
  }
  __nv_bfloat16* out = static_cast<__nv_bfloat16*>(slices);
  if (dt == TK_F64)
    k_oz_scale_slice<double><<<(unsigned)nb, 256, 0, st>>>((const double*)A, rows, cols, ld, EC, RB, cp, ER, out);
  else
    k_oz_scale_slice<float><<<(unsigned)nb, 256, 0, st>>>((const float*)A, rows, cols, ld, EC, RB, cp, ER, out);
  TK_LAUNCH_CHECK();
  return TK_OK;
}

// Column-exponent digits of X stored transposed (the Gram matrix of the sketch): planes of X^T.
static tk_status oz_split_columns(const double* X, int64_t rows, int64_t cols, void* slices, int* E, void* colmax,
                                  cudaStream_t st) {
  const int64_t rp = cdiv(rows, OZ_KPAD) * OZ_KPAD;
  if (cdiv(cols, 32) > 65535) {
    set_error_msg("emulated float64 product: too many columns for the slicing grid");
    return TK_EINVAL;
  }
  TK_TRY(oz_column_exponents(X, TK_F64, rows, cols, cols, E, colmax, nullptr, st));
  const dim3 gt((unsigned)cdiv(rp, 64), (unsigned)cdiv(cols, 32));
  k_oz_slice_t<double><<<gt, dim3(32, 8), 0, st>>>(X, rows, cols, cols, E, rp, static_cast<__nv_bfloat16*>(slices));
  TK_LAUNCH_CHECK();
  return TK_OK;
}

tk_status oz_residual(const OzMat& A, const double* X, int64_t ldx, int64_t M, void* Xslices, int* EX,
                      const double* b, double* R, int64_t ldr, int* err, cudaStream_t st) {
  if (A.m == 0 || M == 0) return TK_OK;
  TK_TRY(oz_split_vectors(X, TK_F64, M, A.n, ldx, A.EC, Xslices, EX, st));
  return launch_oz_tc<OZ_S, 0, false>({A.planes, A.ER, A.m, A.n, false}, Xslices, EX, (int)M, OZ_S, 1, b, R, ldr,
                                      nullptr, err, st);
}

// Split count of a split-K digit product with `tiles` output tiles: the fewest
// waves (1..8) whose last wave is at least 97 % full, so that no SM idles
// through a ragged last wave (e.g. 64 tiles x 5 splits on 304 slots ran 1.05
// waves); at least 256 values of K per split.
int oz_normal_splits(int64_t m, int64_t n, int64_t M, int S) {
  const int nt = oz_tile_n(S, M);
  const int ctas_per_sm = (S == OZ_S || nt == 64) ? 1 : 2;
  const int64_t tiles = std::max<int64_t>(1, cdiv(n, OT_M) * cdiv(M, nt));
  const int64_t slots = 152 * (int64_t)ctas_per_sm;
  const int64_t maxs = std::max<int64_t>(1, cdiv(m, OT_CHUNK));
  int64_t best = 1;
  double best_eff = -1.0;
  for (int64_t w = 1; w <= 8; ++w) {
    const int64_t sp = std::min<int64_t>(cdiv(w * slots, tiles), maxs);
    const int64_t ctas = tiles * sp;
    const double eff = (double)ctas / (double)(cdiv(ctas, slots) * slots);
    if (eff > best_eff + 1e-9) {
      best_eff = eff;
      best = sp;
    }
    if (eff >= 0.97 || sp == maxs) break;
  }
  return (int)std::max<int64_t>({int64_t(1), best, cdiv(m, OT_MAX_KPS)});  // at most 2^27 values of K per split
}

tk_status oz_normal(const OzMat& A, const double* R, int64_t ldr, int64_t M, void* Rslices, int* EX, double* partial,
                    int splits, int* err, cudaStream_t st) {
  if (M == 0 || A.n == 0) return TK_OK;
  TK_TRY(oz_split_vectors(R, TK_F64, M, A.m, ldr, A.ER, Rslices, EX, st));
  return launch_oz_tc<OZ_S, 1, true>({A.planes, A.EC, A.n, A.m, true}, Rslices, EX, (int)M, OZ_S, splits, nullptr,
                                     partial, A.n, nullptr, err, st);
}

template <typename T>
tk_status oz_lsqr_aw(const OzMat& A, const T* W, int64_t ldw, int count, void* Wslices, int* EW, T* U, int64_t ldu,
                     const double* coef, int* err, cudaStream_t st) {
  if (A.m == 0 || count == 0) return TK_OK;
  constexpr int S = oz_digits<T>();
  TK_TRY(oz_split_vectors(W, sizeof(T) == 8 ? TK_F64 : TK_F32, count, A.n, ldw, A.EC, Wslices, EW, st, S));
  return launch_oz_tc<S, 2, false>({A.planes, A.ER, A.m, A.n, false}, Wslices, EW, count, S, 1, nullptr, U, ldu, coef,
                                   err, st);
}

template <typename T>
tk_status oz_lsqr_aw_split(const OzMat& A, const T* W, int64_t ldw, int count, void* Wslices, int* EW, double* partial,
                           int splits, int* err, cudaStream_t st) {
  if (A.m == 0 || count == 0) return TK_OK;
  constexpr int S = oz_digits<T>();
  TK_TRY(oz_split_vectors(W, sizeof(T) == 8 ? TK_F64 : TK_F32, count, A.n, ldw, A.EC, Wslices, EW, st, S));
  return launch_oz_tc<S, 1, false>({A.planes, A.ER, A.m, A.n, false}, Wslices, EW, count, S, splits, nullptr, partial,
                                   A.m, nullptr, err, st);
}

template <typename T>
tk_status oz_lsqr_atu(const OzMat& A, const T* U, int64_t ldu, int count, void* Uslices, int* EU, double* partial,
                      int splits, int* err, cudaStream_t st) {
  if (A.n == 0 || count == 0) return TK_OK;
  constexpr int S = oz_digits<T>();
  TK_TRY(oz_split_vectors(U, sizeof(T) == 8 ? TK_F64 : TK_F32, count, A.m, ldu, A.ER, Uslices, EU, st, S));
  return launch_oz_tc<S, 1, true>({A.planes, A.EC, A.n, A.m, true}, Uslices, EU, count, S, splits, nullptr, partial,
                                  A.n, nullptr, err, st);
}
template tk_status oz_lsqr_aw<float>(const OzMat&, const float*, int64_t, int, void*, int*, float*, int64_t,
                                     const double*, int*, cudaStream_t);
template tk_status oz_lsqr_aw<double>(const OzMat&, const double*, int64_t, int, void*, int*, double*, int64_t,
                                      const double*, int*, cudaStream_t);
template tk_status oz_lsqr_aw_split<double>(const OzMat&, const double*, int64_t, int, void*, int*, double*, int,
                                            int*, cudaStream_t);
template tk_status oz_lsqr_atu<float>(const OzMat&, const float*, int64_t, int, void*, int*, double*, int, int*,
                                      cudaStream_t);
template tk_status oz_lsqr_atu<double>(const OzMat&, const double*, int64_t, int, void*, int*, double*, int, int*,
                                       cudaStream_t);

// Cluster shape of the fused step for n columns: CL CTAs (a power of two, at most 8, so that each
// CTA's share of a band's 128 rows is a multiple of 4) of cpc columns (a multiple of 128, at most
// 256); CL = 0 when n is beyond 8 x 256.
static void fused_shape(int64_t n, int* CL, int* cpc) {
  const int64_t n64 = cdiv(n, OZ_KPAD) * OZ_KPAD;
  const int64_t need = std::max<int64_t>(1, cdiv(n64, 256));
  int cl = 1;
  while (cl < need && cl < 8) cl *= 2;
  const int c = (int)(cdiv(n64, (int64_t)cl * 128) * 128);
  *CL = c <= 256 ? cl : 0;
  *cpc = c;
}

bool oz_fused_supported(int64_t m, int64_t n, int count) {
  int cl = 0, cpc = 0;
  fused_shape(n, &cl, &cpc);
  return cl > 0 && count >= 1 && count <= FU_NT && m >= 1 && m <= INT32_MAX;
}

tk_status oz_lsqr_fused(const OzMat& A, const float* W, int64_t ldw, int count, void* Wslices, int* EW, float* U,
                        int64_t ldu, const double* coef, double* partial, int max_planes, int* planes, int* err,
                        cudaStream_t st) {
  const int64_t m = A.m, n = A.n;
  int CL = 0, cpc = 0;
  fused_shape(n, &CL, &cpc);
  if (!oz_fused_supported(m, n, count) || max_planes < 1) {
    set_error_msg("fused LSQR step: unsupported shape");
    return TK_EINVAL;
  }
  const int64_t n64 = cdiv(n, OZ_KPAD) * OZ_KPAD;
  TK_TRY(oz_split_vectors(W, TK_F32, count, n, ldw, A.EC, Wslices, EW, st, OZ_LSQR_DIGITS));
  CUtensorMap mA, mW;
  TK_TRY(make_slice_map(&mA, A.planes, m, n64, OT_M, OZ_S));
  TK_TRY(make_slice_map(&mW, Wslices, count, n64, FU_NT, OZ_LSQR_DIGITS));
  const size_t smem = sizeof(FuSmem) + 1024;
  TK_CUDA(cudaFuncSetAttribute(k_oz_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)CL;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.blockDim = dim3(256, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // one wave of resident clusters, each looping over its bands (no second wave)
  static int cached[9] = {0};
  if (!cached[CL]) {
    cfg.gridDim = dim3((unsigned)((152 / CL) * CL), 1, 1);
    int nc = 0;
    TK_CUDA(cudaOccupancyMaxActiveClusters(&nc, k_oz_fused, &cfg));
    cached[CL] = nc > 0 ? nc : 1;
  }
  const int64_t bands = cdiv(m, FU_M);
  const int ncl = (int)std::max<int64_t>(1, std::min<int64_t>({(int64_t)cached[CL], bands, (int64_t)max_planes}));
  cfg.gridDim = dim3((unsigned)(ncl * CL), 1, 1);
  TK_CUDA(cudaLaunchKernelEx(&cfg, k_oz_fused, mA, mW, A.ER, A.EC, (const int*)EW, m, n, count, cpc, U, ldu, coef, partial,
                             err));
  TK_LAUNCH_CHECK();
  *planes = ncl;
  return TK_OK;
}

// The level h of M = R^-1 (n a multiple of 64, h of 128): for every pair of diagonal blocks of M that are
// finished, M12 = -M11 (R12 M22), both products from digits (T = double: 8, float64-accurate; T = float: 4,
// the 28-bit rounded operands); Mt = M^T receives its block first.  With R = D U, D its diagonal, M11 is U11^-1
// D^-1 and R12 M22 has rows of the size of D: in the second product the powers of two of D move from one operand
// to the other, so that the digits of a row of M11 are not spent on the range of D (small lambda: 1 .. 1e-5).
template <typename T>
tk_status oz_tri_level(const double* R, int64_t ldr, int64_t rstride, T* M, T* Mt, int64_t ldm, int64_t mstride, int N,
                       int64_t n, int h, void* work, size_t bytes, int* err, cudaStream_t st) {
  constexpr int S = oz_digits<T>();
  constexpr int NT = 32;
  const int pairs = (int)cdiv(n - h, 2 * (int64_t)h);
  if (pairs <= 0) return TK_OK;
  const int64_t batch = (int64_t)N * pairs, rows = batch * h;
  if (batch > 65535 || rows > INT32_MAX || (double)rows * h > 2e9 * OT_M * NT) {
    set_error_msg("triangular inverse: too many blocks for one launch");
    return TK_EINVAL;
  }
  Arena a;
  a.base = static_cast<char*>(work);
  a.cap = bytes;
  __nv_bfloat16* Ps = a.take<__nv_bfloat16>((size_t)S * rows * h);
  __nv_bfloat16* Qs = a.take<__nv_bfloat16>((size_t)S * rows * h);
  int* EP = a.take<int>((size_t)rows);
  int* EQ = a.take<int>((size_t)rows);
  T* Tt = a.take<T>((size_t)rows * h);  // (R12 M22)^T
  int* up = a.take<int>((size_t)N * n);
  int* down = a.take<int>((size_t)N * n);
  if (!a.ok()) return TK_ENOMEM;
  k_oz_diag_exp<<<dim3((unsigned)cdiv(n, 256), (unsigned)N), 256, 0, st>>>(R, ldr, rstride, (int)n, up, down);
  TK_LAUNCH_CHECK();
  CUtensorMap mP, mQ;
  TK_TRY(make_slice_map(&mP, Ps, rows, h, OT_M, S));
  TK_TRY(make_slice_map(&mQ, Qs, rows, h, NT, S));
  const size_t smem = sizeof(OtSmem<S, NT>) + 1024;
  TK_CUDA(cudaFuncSetAttribute(k_oz_tc<S, 3, NT, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const dim3 gs((unsigned)h, (unsigned)batch);
  const OtTiles tl{(uint32_t)(h / OT_M), (uint32_t)(h / NT), (uint32_t)batch};
  const unsigned g = ot_grid<S, NT>(tl);
  const int64_t pr = 2 * (int64_t)h;  // a pair's step along the diagonal
  OtTri t{pairs, 1, h, (int)n, (int64_t)pairs * h * h, (int64_t)h * h, 1.0};
  k_oz_block_rows<double><<<gs, 256, 0, st>>>(R + h, rstride, pr * (ldr + 1), ldr, pairs, h, (int)n, 0, 1, 0,
                                              nullptr, rows, S, EP, Ps);
  TK_LAUNCH_CHECK();
  k_oz_block_rows<T><<<gs, 256, 0, st>>>(Mt + h * (ldm + 1), mstride, pr * (ldm + 1), ldm, pairs, h, (int)n, 1, 1, 1,
                                         nullptr, rows, S, EQ, Qs);
  TK_LAUNCH_CHECK();
  k_oz_tc<S, 3, NT, false, false>
      <<<g, 256, smem, st>>>(mP, mQ, EP, EQ, h, h, h, h, nullptr, Tt, h, nullptr, err, tl, t);
  TK_LAUNCH_CHECK();
  k_oz_block_rows<T><<<gs, 256, 0, st>>>(M, mstride, pr * (ldm + 1), ldm, pairs, h, (int)n, 0, 0, 0, up, rows, S,
                                         EP, Ps);
  TK_LAUNCH_CHECK();
  k_oz_block_rows<T><<<gs, 256, 0, st>>>(Tt, (int64_t)pairs * h * h, (int64_t)h * h, h, pairs, h, (int)n, 1, 0, 0, down,
                                         rows, S, EQ, Qs);
  TK_LAUNCH_CHECK();
  t = OtTri{pairs, 2, h, (int)n, mstride, pr * (ldm + 1), -1.0};
  k_oz_tc<S, 3, NT, false, false>
      <<<g, 256, smem, st>>>(mP, mQ, EP, EQ, h, h, h, h, nullptr, Mt + h * ldm, ldm, nullptr, err, tl, t);
  TK_LAUNCH_CHECK();
  k_oz_block_transpose<T><<<dim3((unsigned)(h / 32), (unsigned)(h / 32), (unsigned)batch), 256, 0, st>>>(
      Mt, M, ldm, mstride, pairs, h, (int)n);
  TK_LAUNCH_CHECK();
  return TK_OK;
}
template tk_status oz_tri_level<float>(const double*, int64_t, int64_t, float*, float*, int64_t, int64_t, int, int64_t,
                                       int, void*, size_t, int*, cudaStream_t);
template tk_status oz_tri_level<double>(const double*, int64_t, int64_t, double*, double*, int64_t, int64_t, int,
                                        int64_t, int, void*, size_t, int*, cudaStream_t);

// Lambdas per pass of the levels: their planes take 16 to 32 bytes per element of a level, and 2 GiB of them are
// thousands of tiles already
template <typename T>
int oz_tri_lambdas(int64_t n, int N, int h0) {
  int64_t most = 1;
  for (int64_t h = h0; h < n; h *= 2)
    most = std::max(most, cdiv(n - h, 2 * h) * h * h * (int64_t)(4 * oz_digits<T>() + sizeof(T)));
  return (int)std::max<int64_t>(1, std::min<int64_t>(N, (int64_t(2) << 30) / most));
}
template int oz_tri_lambdas<float>(int64_t, int, int);
template int oz_tri_lambdas<double>(int64_t, int, int);

template <typename T>
size_t oz_tri_workspace(int64_t n, int N, int h0) {
  size_t most = 0;
  for (int64_t h = h0; h < n; h *= 2) {
    const size_t rows = (size_t)oz_tri_lambdas<T>(n, N, h0) * cdiv(n - h, 2 * h) * h;
    Arena a;
    a.take<__nv_bfloat16>(oz_digits<T>() * rows * h);
    a.take<__nv_bfloat16>(oz_digits<T>() * rows * h);
    a.take<int>(rows);
    a.take<int>(rows);
    a.take<T>(rows * h);
    a.take<int>((size_t)N * n);
    a.take<int>((size_t)N * n);
    most = std::max(most, a.used + 256);
  }
  return most;
}
template size_t oz_tri_workspace<float>(int64_t, int, int);
template size_t oz_tri_workspace<double>(int64_t, int, int);

static int oz_sketch_splits(int64_t L, int64_t c, int64_t s) {
  const int64_t tiles = cdiv(c, OT_M) * cdiv(s, OT_N);
  return tiles >= 152 ? (int)cdiv(L, OT_MAX_KPS) : oz_normal_splits(L, c, s);
}
// Y (+)= sum_z part[z]
__global__ void k_oz_sum_planes(const double* __restrict__ part, int splits, int64_t total, double* __restrict__ Y,
                                int add) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total; k += (int64_t)gridDim.x * blockDim.x) {
    double acc = add ? Y[k] : 0.0;
#pragma unroll 4
    for (int z = 0; z < splits; ++z) acc += part[(int64_t)z * total + k];
    Y[k] = acc;
  }
}

// The columns of the embedding whose float64 values and 8 digit planes (24 bytes a value) are held at a time: 2 GiB of
// them, a product of thousands of values of K for every s, so that the blocks cost nothing to speak of (262144 x 2048,
// s = 8192: 445.8 ms in 25 blocks, 443.4 in one with 48 GiB of scratch; 65536 x 1024, s = 4096: 38.7 and 38.5; on the
// float64 pipe 7361 and 503).
static int64_t oz_sketch_block(int64_t L, int64_t s) {
  const int64_t fit = (int64_t(2) << 30) / (24 * s) / OT_CHUNK * OT_CHUNK;
  return std::min<int64_t>(L, std::max<int64_t>(fit, OT_CHUNK));
}

static void oz_sketch_carve(Arena& a, int64_t L, int64_t c, int64_t s, double** G, void** Gs, int** E, double** part) {
  const int64_t len = oz_sketch_block(L, s);
  const int sp = oz_sketch_splits(len, c, s);
  *G = a.take<double>((size_t)s * len);
  *Gs = a.take<char>(oz_slices_bytes(s, len));
  *E = a.take<int>(s);
  *part = sp > 1 || len < L ? a.take<double>((size_t)sp * s * c) : nullptr;
}

size_t oz_sketch_workspace(int64_t L, int64_t c, int64_t s) {
  Arena a;
  double *G, *part;
  void* Gs;
  int* E;
  oz_sketch_carve(a, L, c, s, &G, &Gs, &E, &part);
  return a.used + 256;
}

tk_status oz_sketch(const OzMat& A, bool under, uint64_t seed, int64_t s, double* Y, void* work, size_t bytes,
                    int* err, cudaStream_t st) {
  const int64_t L = under ? A.n : A.m, c = under ? A.m : A.n;
  if (s == 0 || c == 0) return TK_OK;
  Arena a;
  a.base = static_cast<char*>(work);
  a.cap = bytes;
  double *G, *part;
  void* Gs;
  int* E;
  oz_sketch_carve(a, L, c, s, &G, &Gs, &E, &part);
  if (!a.ok()) return TK_ENOMEM;
  const int64_t block = oz_sketch_block(L, s), n64 = cdiv(A.n, OZ_KPAD) * OZ_KPAD;
  const int sp = oz_sketch_splits(block, c, s);
  double* out = part ? part : Y;
  const __nv_bfloat16* planes = static_cast<const __nv_bfloat16*>(A.planes);
  // blocks of columns of the embedding (rows of A, or its columns where m < n), their products added in order
  for (int64_t k0 = 0; k0 < L; k0 += block) {
    const int64_t len = std::min(block, L - k0);
    TK_TRY(gauss_fill(seed, s, L, k0, len, G, st));
    TK_TRY(oz_split_vectors(G, TK_F64, s, len, len, (under ? A.EC : A.ER) + k0, Gs, E, st));
    if (under)
      TK_TRY((launch_oz_tc<OZ_S, 1, false>({planes + k0, A.ER, A.m, len, false, n64, A.m * n64}, Gs, E, (int)s, OZ_S, sp,
                                           nullptr, out, c, nullptr, err, st)));
    else
      TK_TRY((launch_oz_tc<OZ_S, 1, true>({planes + k0 * n64, A.EC, A.n, len, true, n64, A.m * n64}, Gs, E, (int)s, OZ_S,
                                          sp, nullptr, out, c, nullptr, err, st)));
    if (part) {
      k_oz_sum_planes<<<(unsigned)std::min<int64_t>(cdiv(s * c, 256), 152 * 8), 256, 0, st>>>(part, sp, s * c, Y,
                                                                                             k0 > 0);
      TK_LAUNCH_CHECK();
    }
  }
  return TK_OK;
}

// Splits of the sum over the r rows of Y when the upper triangle's tiles (128 x 32) leave SMs idle.
static int oz_gram_splits(int64_t r, int64_t c) {
  int64_t tiles = 0;
  for (int64_t i = 0; i < cdiv(c, OT_M); ++i) tiles += std::min<int64_t>(cdiv(c, OT_N), cdiv((i + 1) * OT_M, OT_N));
  const int64_t want = tiles >= 152 ? 1 : 152 / tiles, maxs = std::max<int64_t>(1, r / (2 * OT_CHUNK));
  return (int)std::max<int64_t>(std::min(want, maxs), cdiv(r, OT_MAX_KPS));
}

size_t oz_gram_workspace(int64_t r, int64_t c) {
  Arena a;
  a.take<char>(oz_slices_bytes(c, r));
  a.take<int>(c);
  a.take<char>(oz_colmax_bytes(c));
  const int sp = oz_gram_splits(r, c);
  if (sp > 1) a.take<double>((size_t)sp * c * c);
  return a.used + 256;
}

tk_status oz_gram(const double* Y, int64_t r, int64_t c, double* C, void* work, size_t bytes, int* err,
                  cudaStream_t st) {
  if (c == 0) return TK_OK;
  if (r == 0) {
    TK_CUDA(cudaMemsetAsync(C, 0, sizeof(double) * (size_t)c * c, st));
    return TK_OK;
  }
  Arena a;
  a.base = static_cast<char*>(work);
  a.cap = bytes;
  void* Ys = a.take<char>(oz_slices_bytes(c, r));
  int* E = a.take<int>(c);
  void* mx = a.take<char>(oz_colmax_bytes(c));
  const int sp = oz_gram_splits(r, c);
  double* part = sp > 1 ? a.take<double>((size_t)sp * c * c) : nullptr;
  if (!a.ok()) return TK_ENOMEM;
  TK_TRY(oz_split_columns(Y, r, c, Ys, E, mx, st));
  // n = 777, s = 12432: 0.47 ms in one piece on 100 of the 152 SMs, 0.18 in splits
  TK_TRY((launch_oz_tc<OZ_S, 1, false, true>({Ys, E, c, r, false}, Ys, E, (int)c, OZ_S, sp, nullptr, sp > 1 ? part : C,
                                             c, nullptr, err, st)));
  if (sp > 1) {  // (below the diagonal tiles the planes hold nothing: those sums are not read)
    k_oz_sum_planes<<<(unsigned)std::min<int64_t>(cdiv(c * c, 256), 152 * 8), 256, 0, st>>>(part, sp, c * c, C, 0);
    TK_LAUNCH_CHECK();
  }
  return TK_OK;
}

// Lambdas whose panels of 256 rows share a launch: 2 GiB of planes at most
static int oz_panel_lambdas(int64_t np, int N) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(N, (int64_t(2) << 30) / (np * 256 * OZ_S * 2)));
}
// values of a digit plane: of the block rows' planes of 64, or of the panels' of 256
static size_t oz_chol_plane(int64_t np, int N) {
  return (size_t)np * std::max(N * 64, np > 256 ? oz_panel_lambdas(np, N) * 256 : 0);
}

size_t oz_chol_workspace(int64_t np, int N) {
  Arena a;
  a.take<__nv_bfloat16>(OZ_S * oz_chol_plane(np, N));
  a.take<int>((size_t)N * np);
  return a.used + 256;
}

tk_status oz_chol_begin(double* R, int64_t ldr, int64_t rstride, int N, int64_t np, void* work, size_t bytes,
                        int* err, OzCholPlan* plan, cudaStream_t st) {
  if (np % 64 || ldr % 4 || rstride % 4 || (uintptr_t)R % 32 || N > kOzCholLambdas || np > INT32_MAX) {
    set_error_msg("emulated Cholesky: unsupported order or lambda count");
    return TK_EINVAL;
  }
  Arena a;
  a.base = static_cast<char*>(work);
  a.cap = bytes;
  const size_t sb = sizeof(__nv_bfloat16) * (size_t)N * OZ_S * np * 64;
  plan->slices = a.take<__nv_bfloat16>(OZ_S * oz_chol_plane(np, N));
  plan->EC = a.take<int>((size_t)N * np);
  if (!a.ok()) return TK_ENOMEM;
  plan->R = R;
  plan->ldr = ldr;
  plan->rstride = rstride;
  plan->N = N;
  plan->np = np;
  plan->err = err;
  // rows of the slice planes beyond a step's panel width are read by the
  // edge tiles (their products are discarded): keep them finite
  TK_CUDA(cudaMemsetAsync(plan->slices, 0, sb, st));
  EncodeTiledFn fn;
  TK_TRY(encode_fn(&fn));
  const cuuint64_t dims[3] = {64, (cuuint64_t)np, (cuuint64_t)N * OZ_S};
  const cuuint64_t strides[2] = {128, (cuuint64_t)np * 128};
  const cuuint32_t estr[3] = {1, 1, 1};
  for (int which = 0; which < 2; ++which) {
    const cuuint32_t box[3] = {64, which == 0 ? (cuuint32_t)CS_M : (cuuint32_t)CS_N, 1};
    CUresult r = fn(which == 0 ? &plan->mP : &plan->mQ, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, plan->slices, dims,
                    strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
      set_error_msg("cuTensorMapEncodeTiled rejected the panel slice layout");
      return TK_ECUDA;
    }
  }
  TK_CUDA(cudaFuncSetAttribute(k_oz_syrk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(CsSmem) + 1024)));
  if (np > 256) {
    // the same memory, as the planes of a panel of 256 rows
    const int64_t rows = (int64_t)oz_panel_lambdas(np, N) * np;
    if (rows > INT32_MAX - 2 * OT_M || (double)rows * np > 2e9 * OT_M * OT_N) {
      set_error_msg("emulated Cholesky: unsupported order or lambda count");
      return TK_EINVAL;
    }
    TK_TRY(make_slice_map(&plan->mP256, plan->slices, rows, 256, OT_M, OZ_S));
    TK_TRY(make_slice_map(&plan->mQ256, plan->slices, rows, 256, OT_N, OZ_S));
    TK_CUDA(cudaFuncSetAttribute(k_oz_tc<OZ_S, 4, 32, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(sizeof(OtSmem<OZ_S, 32>) + 1024)));
    TK_CUDA(cudaFuncSetAttribute(k_oz_panel256, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPanelSmem));
  }
  return TK_OK;
}

// Right-looking in panels of 4 block rows: after block row kb the rest of its panel (rem rows, all columns
// right of it) takes the product of its 64 rows; after the panel's last one the whole trailing block takes the
// product of the panel's 256 rows.  A trailing element is then read, scaled and written once per 256 rows
// instead of once per 64, which is what bounded the update (the float64 pipe and the integer work of an
// element's flush, not the products): order 4096, 64 lambda 138 ms for all updates of 64 rows, now 73; order
// 2048, 32 lambda 10.3, now 6.7; order 1024, 16 lambda 1.25, now 1.10.
tk_status oz_chol_step(const OzCholPlan& plan, int kb, cudaStream_t st) {
  const int64_t w = plan.np - (int64_t)(kb + 1) * 64;
  if (w <= 0) return TK_OK;
  const int64_t rem = std::min<int64_t>(w, (3 - kb % 4) * 64);
  if (rem == 0) {
    const int kb0 = kb - 3, nl = oz_panel_lambdas(plan.np, plan.N);
    const int64_t rows = (int64_t)nl * plan.np, c0 = (int64_t)(kb + 1) * 64;
    const uint32_t gx = (uint32_t)cdiv(w, OT_M);
    const OtTri t{1, 0, (int)plan.np, (int)w, plan.rstride, 0, 1.0};
    for (int l0 = 0; l0 < plan.N; l0 += nl) {
      const int cnt = std::min(nl, plan.N - l0);
      double* Rl = plan.R + (int64_t)l0 * plan.rstride;
      k_oz_panel256<<<dim3((unsigned)cdiv(w, 32), (unsigned)cnt), 256, kPanelSmem, st>>>(
          Rl, plan.ldr, plan.rstride, plan.np, kb0, rows, static_cast<__nv_bfloat16*>(plan.slices), plan.EC);
      TK_LAUNCH_CHECK();
      const OtTiles tl{gx * (gx + 1) / 2 * 4, 1, (uint32_t)cnt};
      k_oz_tc<OZ_S, 4, 32, false, false>
          <<<ot_grid<OZ_S, 32>(tl), 128 + ot_epi<4>, sizeof(OtSmem<OZ_S, 32>) + 1024, st>>>(
              plan.mP256, plan.mQ256, plan.EC, plan.EC, w, (int)w, 256, 256, nullptr, Rl + c0 * (plan.ldr + 1), plan.ldr,
              nullptr, plan.err, tl, t);
      TK_LAUNCH_CHECK();
    }
    return TK_OK;
  }
  __nv_bfloat16* sl = static_cast<__nv_bfloat16*>(plan.slices);
  k_oz_panel_slice<<<dim3((unsigned)cdiv(w, 32), (unsigned)plan.N), 256, 0, st>>>(plan.R, plan.ldr, plan.rstride,
                                                                                   plan.np, kb, sl, plan.EC);
  TK_LAUNCH_CHECK();
  const dim3 grid((unsigned)cdiv(rem, CS_M), (unsigned)cdiv(w / CS_N, CS_TILES), (unsigned)plan.N);
  k_oz_syrk<<<grid, 384, sizeof(CsSmem) + 1024, st>>>(plan.mP, plan.mQ, plan.EC, plan.np, kb, (int)rem, plan.R,
                                                     plan.ldr, plan.rstride, plan.err);
  TK_LAUNCH_CHECK();
  return TK_OK;
}

}  // namespace tk

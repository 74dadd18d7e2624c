// [~, Sigma, V] = svd(Y, 'econ') of Algorithm 3 step 4 by one-sided Jacobi on
// the rows of Y (the columns of Y^T): the rows are rotated until they are
// orthogonal; their norms are sigma and the normalized rows V.
//
//  * Before the first sweep Y is turned by an orthogonal Q close to its left
//    singular vectors: Q from a QR factorization of C = Y Y^T (one step of the
//    QR algorithm), W = Q Y.  Q only has to be orthogonal (its rows are
//    orthogonalized twice), so the singular values and the accuracy of the
//    rotations are those of Y; sketches need 8 to 10 sweeps from W where they
//    need 16 to 24 from Y.
//  * Rows are paired in blocks of two by the round-robin (circle) schedule: a
//    CTA keeps the four rows of a block pair in registers and rotates the four
//    cross pairs, so a sweep of s rows is about s / 2 launches (the first of
//    them also rotates the pairs inside the blocks).  Sweeps repeat until no
//    pair is rotated.
//
// GB300 issues two float64 FMA per clock and SM, so a warp's float64
// instruction holds the pipe for 16 clocks: the kernels spend few of them
// outside the dot products and rotations (sums fold several values at once,
// rotation angles are taken in float32 -- a rotation by a slightly different
// angle is still a rotation -- and only cos and sin are refined in float64).
// A 462 x 1000 sketch: 217 ms (23 sweeps of 461 launches, a warp per pair) ->
// 30 ms.
#include <algorithm>
#include <numeric>
#include <vector>

#include "tk_lsqr.cuh"

namespace tk {
namespace {

// ---- block pairs ------------------------------------------------------------
// Pair k of round `round` of the circle schedule over sp (even) players.
__device__ __forceinline__ void circle_pair(int64_t sp, int64_t round, int64_t k, int64_t* p, int64_t* q) {
  int64_t a, b;
  if (k == 0) {
    a = sp - 1;
    b = round;
  } else {
    a = (round + k) % (sp - 1);
    b = (round - k + (sp - 1)) % (sp - 1);
  }
  *p = a < b ? a : b;
  *q = a < b ? b : a;
}

struct JacSmem {
  double red[2][16];  // per warp: the two dot products
  double cs[2], sn[2];
  double nr[4];       // squared row norms
  int rot[2];
};

// Rotation that makes rows of squared norms a, b and dot product g orthogonal (rows already orthogonal
// to tol, or one of them zero: false).  t = tan of the angle in float32 from the scaled ratio zeta =
// (b - a) / (2 g): off by 1e-7 relative it leaves 1e-7 of g for the next sweep; the norms' update a - t g is
// exact to second order in that.  Where the ratio leaves float32 (a row of nothing but rounding errors
// against a full one) t = 1 / (2 zeta) with float64's exponent: a t lost to zero would rotate the pair in every sweep.
// cos = (1 + t^2)^(-1/2) by two Newton steps from the float32 value.
__device__ __forceinline__ bool jac_angle(double a, double b, double g, double tol, double* c, double* s, double* t) {
  if (!(a > 0.0) || !(b > 0.0)) return false;
  if (!(g * g > tol * tol * (a * b))) return false;  // (in range: the rows are scaled, see svd_start)
  const double d1 = b - a, d2 = 2.0 * g;
  // both scaled by the power of two that brings the larger to [1, 2): float32 then holds their ratio
  const int e1 = (__double2hiint(d1) >> 20) & 0x7ff, e2 = (__double2hiint(d2) >> 20) & 0x7ff;
  const int e = e1 > e2 ? e1 : e2;
  const double sc = __hiloint2double((e > 2045 ? 1 : 2046 - e) << 20, 0);
  const float f1 = (float)(d1 * sc), f2 = (float)(d2 * sc);
  const float z = f1 / f2, az = fabsf(z);
  const float ta = az > 1e8f ? 0.5f / az : 1.0f / (az + sqrtf(fmaf(az, az, 1.0f)));
  *t = (double)((f1 >= 0.0f) == (f2 >= 0.0f) ? ta : -ta);
  if (az > 1e30f) {  // g / d1 from the float32 quotient of the mantissas (d1 the larger: e == e1)
    const float q = 0.5f * (float)(d2 * __hiloint2double((2046 - e2) << 20, 0)) / f1;
    *t = (double)q * __hiloint2double((1023 + e2 - e1) << 20, 0);
  }
  const double x = fma(*t, *t, 1.0);
  double r = (double)rsqrtf((float)x);
  r = r * fma(-0.5 * x * r, r, 1.5);
  r = r * fma(-0.5 * x * r, r, 1.5);
  *c = r;
  *s = r * *t;
  return true;
}

// The angles of the pairs (A, B) and (C, D) of a block's four rows from the threads' parts g0, g1 of their dot
// products: rotations and flags in S, the norms updated, rotations counted by lanes 0 and 16 of warp 0.
template <int TH, int A, int B, int C, int D>
__device__ __forceinline__ void jac_two_angles(double g0, double g1, double tol, JacSmem& S, int* nrot) {
  constexpr int NW = TH / 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // lanes 0-15 sum g0, lanes 16-31 g1: one exchange, then four steps for both
  const bool up = lane >= 16;
  double v = (up ? g1 : g0) + __shfl_xor_sync(0xffffffffu, up ? g0 : g1, 16);
#pragma unroll
  for (int o = 8; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((lane & 15) == 0) S.red[lane >> 4][w] = v;
  __syncthreads();
  if (w == 0) {
    const int h = lane >> 4;
    double g = (lane & 15) < NW ? S.red[h][lane & 15] : 0.0;
#pragma unroll
    for (int o = NW / 2; o >= 1; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
    const int ra = h ? C : A, rb = h ? D : B;
    const double a = S.nr[ra], b = S.nr[rb];
    double c = 1.0, s = 0.0, t = 0.0;
    const bool rot = jac_angle(a, b, g, tol, &c, &s, &t);
    if ((lane & 15) == 0) {
      S.rot[h] = rot;
      S.cs[h] = c;
      S.sn[h] = s;
      if (rot) {
        S.nr[ra] = a - t * g;
        S.nr[rb] = b + t * g;
        ++*nrot;
      }
    }
  }
  __syncthreads();
}

// The pairs (A, B) and (C, D) of the four rows x[][] held by the block (thread t: values t, t + TH, ..).
template <int NE, int TH, int A, int B, int C, int D>
__device__ __forceinline__ void jac_two_pairs(double (&x)[4][NE], int ne, double tol, JacSmem& S, int* nrot) {
  double g0 = 0.0, g1 = 0.0;
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    if (e < ne) {
      g0 = fma(x[A][e], x[B][e], g0);
      g1 = fma(x[C][e], x[D][e], g1);
    }
  }
  jac_two_angles<TH, A, B, C, D>(g0, g1, tol, S, nrot);
  if (S.rot[0]) {
    const double c = S.cs[0], s = S.sn[0];
#pragma unroll
    for (int e = 0; e < NE; ++e) {
      if (e < ne) {
        const double u = x[A][e], y = x[B][e];
        x[A][e] = c * u - s * y;
        x[B][e] = s * u + c * y;
      }
    }
  }
  if (S.rot[1]) {
    const double c = S.cs[1], s = S.sn[1];
#pragma unroll
    for (int e = 0; e < NE; ++e) {
      if (e < ne) {
        const double u = x[C][e], y = x[D][e];
        x[C][e] = c * u - s * y;
        x[D][e] = s * u + c * y;
      }
    }
  }
}

// The same for rows that stay in memory (x[i]: row i, null if absent): every thread reads and writes its own
// values t, t + TH, .. throughout.
template <int TH>
__device__ __forceinline__ double jac_dot_mem(const double* x, const double* y, int64_t n) {
  double g = 0.0;
  if (x && y) {
#pragma unroll 4
    for (int64_t j = threadIdx.x; j < n; j += TH) g = fma(x[j], y[j], g);
  }
  return g;
}
template <int TH>
__device__ __forceinline__ void jac_rotate_mem(double* x, double* y, int64_t n, double c, double s) {
#pragma unroll 4
  for (int64_t j = threadIdx.x; j < n; j += TH) {
    const double u = x[j], v = y[j];
    x[j] = c * u - s * v;
    y[j] = s * u + c * v;
  }
}
template <int TH, int A, int B, int C, int D>
__device__ __forceinline__ void jac_two_pairs_mem(double* const (&x)[4], int64_t n, double tol, JacSmem& S,
                                                  int* nrot) {
  const double g0 = jac_dot_mem<TH>(x[A], x[B], n), g1 = jac_dot_mem<TH>(x[C], x[D], n);
  jac_two_angles<TH, A, B, C, D>(g0, g1, tol, S, nrot);
  if (S.rot[0]) jac_rotate_mem<TH>(x[A], x[B], n, S.cs[0], S.sn[0]);  // (an absent row has norm 0: no rotation)
  if (S.rot[1]) jac_rotate_mem<TH>(x[C], x[D], n, S.cs[1], S.sn[1]);
}

// A row of less than 2^-106 = (2^-53)^2 of the largest norm, which is scaled to 1, counts as zero: it is what rounding
// left of a row that depends on others, and each sweep would rotate the rounding errors of the sweep before (16 rows
// with 6 nonzero columns: the cap of 80 sweeps, now 19).
__device__ __forceinline__ double jac_norm2(double nrm2) { return nrm2 > 0x1p-212 ? nrm2 : 0.0; }

// Block pair k of a round: rows 2p, 2p + 1 and 2q, 2q + 1 of W (rows >= s: absent, norm 0).  first:
// also the pairs inside the two blocks (once a sweep).
template <int NE, int TH>
__device__ __forceinline__ void jac_block_pair(double* __restrict__ W, double* __restrict__ nrm2, int64_t s,
                                               int64_t n, int64_t sp, int64_t round, int64_t k, double tol,
                                               int* __restrict__ rotated, JacSmem& S) {
  int64_t p, q;
  circle_pair(sp, round, k, &p, &q);
  const bool first = round == 0;
  const int64_t r[4] = {2 * p, 2 * p + 1, 2 * q, 2 * q + 1};
  if (!first && r[2] >= s) return;  // pair with the dummy block
  const int ne = (int)((n + TH - 1) / TH);
  double x[4][NE];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int e = 0; e < NE; ++e) {
      const int64_t j = threadIdx.x + (int64_t)TH * e;
      x[i][e] = (r[i] < s && j < n) ? W[r[i] * n + j] : 0.0;
    }
  if (threadIdx.x < 4) S.nr[threadIdx.x] = jac_norm2(r[threadIdx.x] < s ? nrm2[r[threadIdx.x]] : 0.0);
  __syncthreads();
  int nrot = 0;
  if (first) jac_two_pairs<NE, TH, 0, 1, 2, 3>(x, ne, tol, S, &nrot);
  jac_two_pairs<NE, TH, 0, 2, 1, 3>(x, ne, tol, S, &nrot);
  jac_two_pairs<NE, TH, 0, 3, 1, 2>(x, ne, tol, S, &nrot);
  // warp 0's lanes 0 and 16 counted their own pair's rotations; the block writes back if there were any
  const int any = __syncthreads_or(nrot);
  if (!any) return;
  if (nrot) atomicAdd(rotated, nrot);
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int e = 0; e < NE; ++e) {
      const int64_t j = threadIdx.x + (int64_t)TH * e;
      if (r[i] < s && j < n) W[r[i] * n + j] = x[i][e];
    }
  if (threadIdx.x < 4 && r[threadIdx.x] < s) nrm2[r[threadIdx.x]] = S.nr[threadIdx.x];
}

// The same with the rows in memory, for any n: bound as the register form by its chain of dot products and angles, the
// rows read from L2 for each of them (66 x 8200, 9 sweeps: 24.5 ms, in registers 66 x 8192 26.1; 200 x 16000: 111 ms; a
// warp per pair of rows, as it was once, 55 and 361).
template <int TH>
__device__ __forceinline__ void jac_block_pair_mem(double* __restrict__ W, double* __restrict__ nrm2, int64_t s,
                                                   int64_t n, int64_t sp, int64_t round, int64_t k, double tol,
                                                   int* __restrict__ rotated, JacSmem& S) {
  int64_t p, q;
  circle_pair(sp, round, k, &p, &q);
  const bool first = round == 0;
  const int64_t r[4] = {2 * p, 2 * p + 1, 2 * q, 2 * q + 1};
  if (!first && r[2] >= s) return;  // pair with the dummy block
  double* x[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) x[i] = r[i] < s ? W + r[i] * n : nullptr;
  if (threadIdx.x < 4) S.nr[threadIdx.x] = jac_norm2(r[threadIdx.x] < s ? nrm2[r[threadIdx.x]] : 0.0);
  __syncthreads();
  int nrot = 0;
  if (first) jac_two_pairs_mem<TH, 0, 1, 2, 3>(x, n, tol, S, &nrot);
  jac_two_pairs_mem<TH, 0, 2, 1, 3>(x, n, tol, S, &nrot);
  jac_two_pairs_mem<TH, 0, 3, 1, 2>(x, n, tol, S, &nrot);
  if (nrot) atomicAdd(rotated, nrot);
  if (threadIdx.x < 4 && r[threadIdx.x] < s) nrm2[r[threadIdx.x]] = S.nr[threadIdx.x];
}

// One round of every matrix: CTA = (matrix, block pair).
struct SvdDesc {
  double* W;
  double* nrm2;
  int64_t s, n, sp;  // sp: blocks of two rows, rounded up to an even count
  int* rotated;
  int done;
};
struct SvdTile {
  int job, k;
};
template <int NE, int TH>
__global__ void __launch_bounds__(TH)
    k_jacobi_round(const SvdDesc* __restrict__ D, const SvdTile* __restrict__ tl, int64_t round, double tol) {
  __shared__ JacSmem S;
  const SvdTile t = tl[blockIdx.x];
  const SvdDesc& d = D[t.job];
  if (d.done || round >= d.sp - 1) return;
  jac_block_pair<NE, TH>(d.W, d.nrm2, d.s, d.n, d.sp, round, t.k, tol, d.rotated, S);
}
template <int TH>
__global__ void __launch_bounds__(TH)
    k_jacobi_round_mem(const SvdDesc* __restrict__ D, const SvdTile* __restrict__ tl, int64_t round, double tol) {
  __shared__ JacSmem S;
  const SvdTile t = tl[blockIdx.x];
  const SvdDesc& d = D[t.job];
  if (d.done || round >= d.sp - 1) return;
  jac_block_pair_mem<TH>(d.W, d.nrm2, d.s, d.n, d.sp, round, t.k, tol, d.rotated, S);
}

// Squared row norms at the start of a sweep (a warp to each of the block pair's four rows).
__global__ void __launch_bounds__(128) k_jacobi_norms(const SvdDesc* __restrict__ D, const SvdTile* __restrict__ tl) {
  const SvdTile t = tl[blockIdx.x];
  const SvdDesc& d = D[t.job];
  const int64_t r = 4 * (int64_t)t.k + (threadIdx.x >> 5);
  if (t.k == 0 && threadIdx.x == 0 && !d.done) *d.rotated = 0;
  if (d.done || r >= d.s) return;
  const int lane = threadIdx.x & 31;
  double a = 0.0;
#pragma unroll 4
  for (int64_t i = lane; i < d.n; i += 32) a = fma(d.W[r * d.n + i], d.W[r * d.n + i], a);
  a = warp_sum(a);
  if (lane == 0) d.nrm2[r] = a;
}

__global__ void k_row_norms(const double* __restrict__ W, int64_t n, double* __restrict__ nrm) {
  __shared__ double sh[32];
  const int64_t p = blockIdx.x;
  double a = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) a = fma(W[p * n + i], W[p * n + i], a);
  a = block_sum(a, sh);
  if (threadIdx.x == 0) nrm[p] = sqrt(a);
}

// V[k*s + j] = W[perm[j]][k] / nrm[perm[j]] ; sigma[j] = nrm[perm[j]] / scale.  32 x 32 tiles through shared memory:
// rows of W are read and rows of V written contiguously.
__global__ void __launch_bounds__(256)
    k_write_v(const double* __restrict__ W, const double* __restrict__ nrm, const int* __restrict__ perm, int64_t s,
              int64_t n, const double* __restrict__ scale, double* __restrict__ V, double* __restrict__ sigma) {
  __shared__ double tile[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t k0 = (int64_t)blockIdx.x * 32, j0 = (int64_t)blockIdx.y * 32;
  for (int r = ty; r < 32; r += 8) {
    const int64_t j = j0 + r, k = k0 + tx;
    if (j < s && k < n) {
      const int p = perm[j];
      const double sg = nrm[p];
      tile[r][tx] = W[(int64_t)p * n + k] * (sg > 0.0 ? 1.0 / sg : 0.0);
      if (blockIdx.x == 0 && tx == 0) sigma[j] = sg / *scale;
    }
  }
  __syncthreads();
  for (int r = ty; r < 32; r += 8) {
    const int64_t k = k0 + r, j = j0 + tx;
    if (j < s && k < n) V[k * s + j] = tile[tx][r];
  }
}

// ---- the orthogonal start -----------------------------------------------------
// Rows of X (s x s, in place) orthonormalized: panels of up to 16 rows, each projected against the
// finished rows and orthogonalized inside (modified Gram-Schmidt), twice.
constexpr int kGsPanel = 16;

// *scale = the power of two that brings the largest of nrm[0 .. s) to [1, 2) (1 if they are zero or not finite); one
// block.
__global__ void __launch_bounds__(256) k_svd_scale(const double* __restrict__ nrm, int64_t s,
                                                   double* __restrict__ scale) {
  __shared__ double sh[8];
  double mx = 0.0;
  for (int64_t i = threadIdx.x; i < s; i += blockDim.x) mx = fmax(mx, nrm[i]);
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) mx = fmax(mx, sh[w]);
    const int e = (__double2hiint(mx) >> 20) & 0x7ff;
    *scale = e > 0 && e < 2046 ? __hiloint2double((2046 - e) << 20, 0) : 1.0;
  }
}
// W = scale Y (Y may be W)
__global__ void k_svd_scaled(const double* Y, int64_t total, const double* __restrict__ scale, double* W) {
  const double sc = *scale;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total; k += (int64_t)gridDim.x * blockDim.x)
    W[k] = sc * Y[k];
}

// X = C + noise of 2^-50 of sqrt(C_ii C_jj): rows of C that are dependent in float64 keep a direction of
// their own (its choice is free), so that Q is a complete basis whatever the rank.  Times scale^2, so that the
// squares of X, fourth powers of Y, stay in float64's range.
__global__ void k_gs_noise(const double* __restrict__ C, int64_t s, const double* __restrict__ scale,
                           double* __restrict__ X) {
  const int64_t i = blockIdx.y;
  const double sc = *scale;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < s; j += (int64_t)gridDim.x * blockDim.x) {
    const uint4 r = philox((uint64_t)(i * s + j), 7u, 0x5eedull);
    const double u = ((double)(int)r.x) * 0x1p-31;  // in [-1, 1)
    X[i * s + j] = sc * (sc * fma(u * 0x1p-50, sqrt(C[i * s + i]) * sqrt(C[j * s + j]), C[i * s + j]));
  }
}

// H[i][q] = X_i . Q_q for the panel's rows i (8 of them per CTA: blockIdx.y) and finished rows q (a warp each).
__global__ void __launch_bounds__(128)
    k_gs_dot(const double* __restrict__ X, int pb, const double* __restrict__ Q, int64_t nq, int64_t s,
             double* __restrict__ H) {
  const int lane = threadIdx.x & 31;
  const int64_t q = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  if (q >= nq) return;
  const int i0 = blockIdx.y * 8;
  double acc[8] = {};
#pragma unroll 2
  for (int64_t c = lane; c < s; c += 32) {
    const double v = Q[q * s + c];
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (i0 + i < pb) acc[i] = fma(X[(int64_t)(i0 + i) * s + c], v, acc[i]);
  }
  int base = 0;
  // halving exchanges: 8 values over the warp, then plain steps
#pragma unroll
  for (int o = 16, nv = 8; o >= 1; o >>= 1) {
    if (nv > 1) {
      const int half = nv / 2;
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k < half) {
          const double send = up ? acc[k] : acc[k + half], keep = up ? acc[k + half] : acc[k];
          acc[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      if (up) base += half;
      nv = half;
    } else {
      acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
    }
  }
  if ((lane & 3) == 0 && i0 + base < pb) H[(int64_t)(i0 + base) * s + q] = acc[0];
}

// X_i -= sum_q H[i][q] Q_q: CTA = row i (blockIdx.y) x 32 columns, 8 groups of finished rows.
__global__ void __launch_bounds__(256)
    k_gs_update(double* __restrict__ X, const double* __restrict__ Q, int64_t nq, int64_t s,
                const double* __restrict__ H) {
  __shared__ double sh[8][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t i = blockIdx.y, c = (int64_t)blockIdx.x * 32 + tx;
  double acc = 0.0;
  if (c < s) {
    const double* h = H + i * s;
#pragma unroll 4
    for (int64_t q = ty; q < nq; q += 8) acc = fma(h[q], Q[q * s + c], acc);
  }
  sh[ty][tx] = acc;
  __syncthreads();
  if (ty == 0 && c < s) {
#pragma unroll
    for (int k = 1; k < 8; ++k) acc += sh[k][tx];
    X[i * s + c] -= acc;
  }
}

// Modified Gram-Schmidt of the panel's rows, in shared memory (pb x s doubles): step j forms the dot
// products of row j with the rows j .. pb - 1 in one reduction, then normalizes row j and subtracts it.
__global__ void __launch_bounds__(128) k_gs_panel(double* __restrict__ X, int pb, int64_t s) {
  extern __shared__ double gs_x[];
  __shared__ double red[4][kGsPanel];
  __shared__ double g[kGsPanel];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t k = threadIdx.x; k < pb * s; k += blockDim.x) gs_x[k] = X[k];
  __syncthreads();
  for (int j = 0; j < pb; ++j) {
    double acc[kGsPanel];
#pragma unroll
    for (int k = 0; k < kGsPanel; ++k) acc[k] = 0.0;
    for (int64_t c = threadIdx.x; c < s; c += blockDim.x) {
      const double v = gs_x[j * s + c];
#pragma unroll
      for (int k = 0; k < kGsPanel; ++k)
        if (k >= j && k < pb) acc[k] = fma(v, gs_x[k * s + c], acc[k]);
    }
    int base = 0;
#pragma unroll
    for (int o = 16, nv = kGsPanel; o >= 1; o >>= 1) {
      if (nv > 1) {
        const int half = nv / 2;
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < kGsPanel / 2; ++k)
          if (k < half) {
            const double send = up ? acc[k] : acc[k + half], keep = up ? acc[k + half] : acc[k];
            acc[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
          }
        if (up) base += half;
        nv = half;
      } else {
        acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
      }
    }
    if ((lane & 1) == 0) red[w][base] = acc[0];
    __syncthreads();
    if (threadIdx.x < kGsPanel)
      g[threadIdx.x] = red[0][threadIdx.x] + red[1][threadIdx.x] + red[2][threadIdx.x] + red[3][threadIdx.x];
    __syncthreads();
    const double gj = g[j];
    const double inv = gj > 0.0 ? rsqrt(gj) : 0.0, inv2 = inv * inv;
    for (int64_t c = threadIdx.x; c < s; c += blockDim.x) {
      const double v = gs_x[j * s + c];
#pragma unroll
      for (int k = 0; k < kGsPanel; ++k)
        if (k > j && k < pb) gs_x[k * s + c] = fma(-g[k] * inv2, v, gs_x[k * s + c]);
      gs_x[j * s + c] = v * inv;
    }
    __syncthreads();
  }
  for (int64_t k = threadIdx.x; k < pb * s; k += blockDim.x) X[k] = gs_x[k];
}

constexpr size_t kGsSmemCap = 200 * 1024;
// rows of a panel whose pb x s doubles fit in shared memory (3 at the largest supported s)
int gs_panel_rows(int64_t s) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(kGsPanel, (int64_t)(kGsSmemCap / (sizeof(double) * s))));
}

// Buffers of one SVD, carved from its scratch.
struct SvdBufs {
  double *W, *nrm, *nrm2, *scale, *C, *Q, *H;
  int *perm, *rotated;
  SvdDesc* desc;
  SvdTile* tiles;
};
// Small matrices start from Y itself: their sweeps are a few dozen launches.  So do those of which not one row of
// s values fits in the shared memory of the panels' Gram-Schmidt.
bool svd_orthogonal_start(int64_t s) { return s >= 64 && s <= (int64_t)(kGsSmemCap / sizeof(double)); }
int64_t block_players(int64_t s) {
  const int64_t nb = cdiv(s, 2);
  return nb + (nb & 1);
}
int64_t svd_tile_count(int64_t s) { return std::max<int64_t>(block_players(s) / 2, 1); }

void svd_carve(Arena& a, int64_t s, int64_t n, SvdBufs& B) {
  B = SvdBufs{};
  B.W = a.take<double>((size_t)s * n);
  B.nrm = a.take<double>((size_t)s);
  B.nrm2 = a.take<double>((size_t)s);
  B.perm = a.take<int>((size_t)s);
  B.scale = a.take<double>(1);
  B.rotated = a.take<int>(1);
  B.desc = a.take<SvdDesc>(1);
  B.tiles = a.take<SvdTile>((size_t)svd_tile_count(s));
  if (svd_orthogonal_start(s)) {
    B.C = a.take<double>((size_t)s * s);
    B.Q = a.take<double>((size_t)s * s);
    B.H = a.take<double>((size_t)kGsPanel * s);
  }
}

// W = scale Q Y (or scale Y), scale the power of two that brings the largest row norm of Y to [1, 2): squares of the
// rotations' dot products and products of squared norms, fourth powers of the rows, leave float64's range for norms
// of 1e-81 or 1e77 otherwise.  svd_finish divides sigma by it.
tk_status svd_start(const double* Y, int64_t s, int64_t n, const SvdBufs& B, cudaStream_t st) {
  k_row_norms<<<(unsigned)s, 256, 0, st>>>(Y, n, B.nrm);
  TK_LAUNCH_CHECK();
  k_svd_scale<<<1, 256, 0, st>>>(B.nrm, s, B.scale);
  TK_LAUNCH_CHECK();
  const unsigned gw = (unsigned)std::min<int64_t>(cdiv(s * n, 256), 152 * 8);
  if (!svd_orthogonal_start(s)) {
    k_svd_scaled<<<gw, 256, 0, st>>>(Y, s * n, B.scale, B.W);
    TK_LAUNCH_CHECK();
    return TK_OK;
  }
  TK_TRY((gemm<double, double, double>(false, true, s, s, n, Y, n, Y, n, B.C, s, 1.0, nullptr, nullptr, 0, st)));
  k_gs_noise<<<dim3((unsigned)cdiv(s, 256), (unsigned)s), 256, 0, st>>>(B.C, s, B.scale, B.Q);
  TK_LAUNCH_CHECK();
  const int pr = gs_panel_rows(s);
  TK_CUDA(cudaFuncSetAttribute(k_gs_panel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGsSmemCap));
  for (int64_t j = 0; j < s; j += pr) {
    const int pb = (int)std::min<int64_t>(pr, s - j);
    double* X = B.Q + j * s;
    for (int pass = 0; pass < 2; ++pass) {
      if (j > 0) {
        k_gs_dot<<<dim3((unsigned)cdiv(j, 4), (unsigned)cdiv(pb, 8)), 128, 0, st>>>(X, pb, B.Q, j, s, B.H);
        TK_LAUNCH_CHECK();
        k_gs_update<<<dim3((unsigned)cdiv(s, 32), (unsigned)pb), 256, 0, st>>>(X, B.Q, j, s, B.H);
        TK_LAUNCH_CHECK();
      }
      k_gs_panel<<<1, 128, sizeof(double) * (size_t)pb * s, st>>>(X, pb, s);
      TK_LAUNCH_CHECK();
    }
  }
  TK_TRY((gemm<double, double, double>(false, false, s, n, s, B.Q, s, Y, n, B.W, n, 1.0, nullptr, nullptr, 0, st)));
  k_svd_scaled<<<gw, 256, 0, st>>>(B.W, s * n, B.scale, B.W);
  TK_LAUNCH_CHECK();
  return TK_OK;
}

// Registers hold 4 rows of a block pair: NE values per thread and row, up to 16 x 512 = 8192 (the largest short
// dimension of a solve).  Longer rows (the SVD called on its own) stay in memory.
tk_status launch_round(int64_t max_n, unsigned tiles, const SvdDesc* dd, const SvdTile* dt, int64_t round, double tol,
                       cudaStream_t st) {
  if (max_n <= 512) k_jacobi_round<4, 128><<<tiles, 128, 0, st>>>(dd, dt, round, tol);
  else if (max_n <= 1024) k_jacobi_round<8, 128><<<tiles, 128, 0, st>>>(dd, dt, round, tol);
  else if (max_n <= 2048) k_jacobi_round<16, 128><<<tiles, 128, 0, st>>>(dd, dt, round, tol);
  else if (max_n <= 4096) k_jacobi_round<16, 256><<<tiles, 256, 0, st>>>(dd, dt, round, tol);
  else if (max_n <= 8192) k_jacobi_round<16, 512><<<tiles, 512, 0, st>>>(dd, dt, round, tol);
  else k_jacobi_round_mem<512><<<tiles, 512, 0, st>>>(dd, dt, round, tol);
  TK_LAUNCH_CHECK();
  return TK_OK;
}

// The sorted singular values and right singular vectors from the rotated
// rows: sigma_j = ||W_perm[j]|| / scale, V[:, j] = W_perm[j] / ||W_perm[j]||.
tk_status svd_finish(const double* W, int64_t s, int64_t n, double* nrm, int* perm, const double* scale,
                     double* sigma, double* V, cudaStream_t st) {
  k_row_norms<<<(unsigned)s, 256, 0, st>>>(W, n, nrm);
  TK_LAUNCH_CHECK();
  std::vector<double> h(s);
  TK_CUDA(cudaMemcpyAsync(h.data(), nrm, sizeof(double) * s, cudaMemcpyDeviceToHost, st));
  TK_CUDA(cudaStreamSynchronize(st));
  std::vector<int> order(s);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return h[a] > h[b]; });
  TK_CUDA(cudaMemcpyAsync(perm, order.data(), sizeof(int) * s, cudaMemcpyHostToDevice, st));
  const dim3 g((unsigned)cdiv(n, 32), (unsigned)cdiv(s, 32));
  k_write_v<<<g, 256, 0, st>>>(W, nrm, perm, s, n, scale, V, sigma);
  TK_LAUNCH_CHECK();
  TK_CUDA(cudaStreamSynchronize(st));  // `order` is a host temporary
  return TK_OK;
}

// Sweeps over all matrices together (one launch per round) until none rotates; sweeps[j] receives the
// count of matrix j.  dd, dt: device copies of hd and of the tiles are made here.
tk_status run_sweeps(std::vector<SvdDesc>& hd, SvdDesc* dd, SvdTile* dt, int* rots, std::vector<int>& sweeps,
                     cudaStream_t st) {
  const int J = (int)hd.size();
  std::vector<SvdTile> tiles;
  int64_t max_rounds = 0, max_n = 0;
  sweeps.assign(J, 0);
  for (int j = 0; j < J; ++j) {
    for (int64_t k = 0; k < svd_tile_count(hd[j].s); ++k) tiles.push_back(SvdTile{j, (int)k});
    if (!hd[j].done) {
      max_rounds = std::max(max_rounds, hd[j].sp - 1);
      max_n = std::max(max_n, hd[j].n);
    }
  }
  TK_CUDA(cudaMemcpyAsync(dd, hd.data(), sizeof(SvdDesc) * J, cudaMemcpyHostToDevice, st));
  TK_CUDA(cudaMemcpyAsync(dt, tiles.data(), sizeof(SvdTile) * tiles.size(), cudaMemcpyHostToDevice, st));
  const double tol = 1e-15;
  const int max_sweeps = 80;
  std::vector<int> hrot(J);
  for (int sweep = 0; sweep < max_sweeps && max_rounds > 0; ++sweep) {
    k_jacobi_norms<<<(unsigned)tiles.size(), 128, 0, st>>>(dd, dt);
    TK_LAUNCH_CHECK();
    for (int64_t r = 0; r < max_rounds; ++r) TK_TRY(launch_round(max_n, (unsigned)tiles.size(), dd, dt, r, tol, st));
    TK_CUDA(cudaMemcpyAsync(hrot.data(), rots, sizeof(int) * J, cudaMemcpyDeviceToHost, st));
    TK_CUDA(cudaStreamSynchronize(st));
    max_rounds = 0;
    for (int j = 0; j < J; ++j) {
      if (hd[j].done) continue;
      sweeps[j] = sweep + 1;
      if (hrot[j] == 0) hd[j].done = 1;
      else max_rounds = std::max(max_rounds, hd[j].sp - 1);
    }
    if (max_rounds > 0) TK_CUDA(cudaMemcpyAsync(dd, hd.data(), sizeof(SvdDesc) * J, cudaMemcpyHostToDevice, st));
  }
  TK_CUDA(cudaStreamSynchronize(st));  // hd and tiles are host memory
  return TK_OK;
}

}  // namespace

size_t svd_workspace(int64_t s, int64_t n) {
  Arena a;
  SvdBufs B;
  svd_carve(a, s, n, B);
  return a.used + 512;
}

tk_status jacobi_svd(const double* Y, int64_t s, int64_t n, double* sigma, double* V, int* sweeps_host, Arena& ar,
                     cudaStream_t st) {
  SvdBufs B;
  svd_carve(ar, s, n, B);
  if (!ar.ok()) return TK_ENOMEM;
  if (s == 0) return TK_OK;
  TK_TRY(svd_start(Y, s, n, B, st));
  std::vector<SvdDesc> hd(1, SvdDesc{B.W, B.nrm2, s, n, block_players(s), B.rotated, s <= 1 ? 1 : 0});
  std::vector<int> sweeps;
  TK_TRY(run_sweeps(hd, B.desc, B.tiles, B.rotated, sweeps, st));
  if (sweeps_host) *sweeps_host = std::max(sweeps[0], 1);
  return svd_finish(B.W, s, n, B.nrm, B.perm, B.scale, sigma, V, st);
}

tk_status jacobi_svd_begin(SvdJob& q, cudaStream_t st) {
  Arena sa;
  sa.base = (char*)q.scratch;
  sa.cap = q.scratch_bytes;
  SvdBufs B;
  svd_carve(sa, q.s, q.n, B);
  if (!sa.ok()) return TK_ENOMEM;
  return q.s > 0 ? svd_start(q.Y, q.s, q.n, B, st) : TK_OK;
}

tk_status jacobi_svd_grouped(std::vector<SvdJob>& jobs, void* work, size_t work_bytes, cudaStream_t st) {
  const int J = (int)jobs.size();
  if (J == 0) return TK_OK;
  std::vector<SvdDesc> hd(J);
  std::vector<SvdBufs> bufs(J);
  Arena a;
  a.base = (char*)work;
  a.cap = work_bytes;
  SvdDesc* dd = a.take<SvdDesc>(J);
  int* rots = a.take<int>(J);
  size_t ntiles = 0;
  for (const auto& j : jobs) ntiles += (size_t)svd_tile_count(j.s);
  SvdTile* dt = a.take<SvdTile>(std::max<size_t>(ntiles, 1));
  if (!a.ok()) {
    set_error_msg("grouped SVD: workspace too small");
    return TK_ENOMEM;
  }
  for (int j = 0; j < J; ++j) {
    SvdJob& q = jobs[j];
    Arena sa;
    sa.base = (char*)q.scratch;
    sa.cap = q.scratch_bytes;
    svd_carve(sa, q.s, q.n, bufs[j]);
    if (!sa.ok()) return TK_ENOMEM;
    hd[j] = SvdDesc{bufs[j].W, bufs[j].nrm2, q.s, q.n, block_players(q.s), rots + j, q.s <= 1 ? 1 : 0};
  }
  std::vector<int> sweeps;
  TK_TRY(run_sweeps(hd, dd, dt, rots, sweeps, st));
  for (int j = 0; j < J; ++j) {
    SvdJob& q = jobs[j];
    q.sweeps = sweeps[j];
    if (q.s > 0) TK_TRY(svd_finish(bufs[j].W, q.s, q.n, bufs[j].nrm, bufs[j].perm, bufs[j].scale, q.sigma, q.V,
                                 st));
  }
  return TK_OK;
}

size_t svd_grouped_workspace(const std::vector<SvdJob>& jobs) {
  Arena a;
  size_t ntiles = 0;
  for (const auto& j : jobs) ntiles += (size_t)svd_tile_count(j.s);
  a.take<SvdDesc>(std::max<size_t>(jobs.size(), 1));
  a.take<int>(std::max<size_t>(jobs.size(), 1));
  a.take<SvdTile>(std::max<size_t>(ntiles, 1));
  return a.used + 1024;
}

}  // namespace tk

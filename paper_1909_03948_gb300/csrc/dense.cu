// dense.cu -- FP64 tall-skinny and small dense linear algebra of the
// randomized eigensolver (Algorithms 2-4) and the low-rank sampling update.
//
//   gram          G = X^T Y (n x s1, n x s2), tiled, deterministic two-stage sum
//   gemm_nn       Y = alpha X S + beta Y (X: n x s1, S: s1 x s2)
//   thin_qr       orthonormal Z with range(Z) = range(Y), the thin-QR step of
//                 PreCholQR (Algorithm 4): shifted Cholesky QR in three passes
//   cgs2_qr       the same by classical Gram-Schmidt with one full
//                 re-orthogonalisation per column ("twice is enough"), the
//                 fallback for a rank-deficient block
//   small_cholesky, trsm_right_upper   R_Z = chol(Z^T Zb), Q = Z R_Z^{-1}
//   small_symeig  cyclic Jacobi with a round-robin parallel ordering, sorted
//                 descending (Algorithm 2: T = S Lambda S^T), A in shared memory up
//                 to 160 x 160 (and V with it up to 90 x 90)
// GB300's FP64 rate is low (a few percent of FP32), so these are written as
// plain FP64 FMA kernels; they are a small share of the eigensolver's time,
// which is dominated by the 2(k+p) Hessian actions.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>
#include <vector>

#include "dfloat.cuh"
#include "internal.h"

namespace hp {

constexpr int GT = 32;  // gram tile

__global__ void k_gram_partial(const double *__restrict__ X, long ldx, int s1, const double *__restrict__ Y, long ldy,
                               int s2, long n, long rows_per_chunk, double *__restrict__ part) {
  __shared__ double xs[GT][GT + 1], ys[GT][GT + 1];
  const int ta = blockIdx.x, tb = blockIdx.y, ch = blockIdx.z;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
  const long r0 = ch * rows_per_chunk, r1 = std::min<long>(n, r0 + rows_per_chunk);
  double acc[4] = {0, 0, 0, 0};
  for (long rb = r0; rb < r1; rb += GT) {
    for (int k = ty; k < GT; k += 8) {
      const long row = rb + tx;
      const int ca = ta * GT + k, cb = tb * GT + k;
      xs[k][tx] = (row < r1 && ca < s1) ? X[ldx * ca + row] : 0.0;
      ys[k][tx] = (row < r1 && cb < s2) ? Y[ldy * cb + row] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int rr = 0; rr < GT; ++rr) {
      const double yv = ys[tx][rr];
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] += xs[ty + 8 * q][rr] * yv;
    }
    __syncthreads();
  }
  const int nta = gridDim.x, ntb = gridDim.y;
  for (int q = 0; q < 4; ++q) {
    const int a = ty + 8 * q, b = tx;
    part[(((long)ch * nta + ta) * ntb + tb) * GT * GT + a * GT + b] = acc[q];
  }
}

// The same partial Gram in double-float arithmetic on the FP32 pipe: the FP64 tiles are
// split into pairs as they are loaded into shared memory (bit manipulation), each thread
// keeps compensated (Dot2) sums for its 4 entries over the chunk's rows, and the chunk's
// entries are stored as doubles.  With sym (X = Y) only the tiles on and above the
// diagonal are formed; k_gram_final mirrors the others.  The compensated sum over a chunk
// is more accurate than FP64 accumulation of the same products (about 2^-48 of the result
// plus n 2^-96 of the terms' magnitudes).
// The next rows are under way while the current ones are multiplied, and a warp leaves out the
// columns beyond s1: 65^3 rows, 100 x 64: 1,750 -> 1,300 us (FP32 pipe: 613 us).
__global__ void k_gram_partial_df(const double *__restrict__ X, long ldx, int s1, const double *__restrict__ Y,
                                  long ldy, int s2, long n, long rows_per_chunk, int sym, double *__restrict__ part) {
  __shared__ float2 xs[GT][GT + 1], ys[GT][GT + 1];
  const int ta = blockIdx.x, tb = blockIdx.y, ch = blockIdx.z;
  if (sym && ta > tb) return;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
  const long r0 = ch * rows_per_chunk, r1 = std::min<long>(n, r0 + rows_per_chunk);
  Dot2 acc[4];
  double xd[4], yd[4];
  auto fetch = [&](long rb) {
    const long row = rb + tx;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int ca = ta * GT + ty + 8 * q, cb = tb * GT + ty + 8 * q;
      xd[q] = (row < r1 && ca < s1) ? X[ldx * ca + row] : 0.0;
      yd[q] = (row < r1 && cb < s2) ? Y[ldy * cb + row] : 0.0;
    }
  };
  auto rows = [&](auto nq) {  // the first nq of this warp's four columns of X
#pragma unroll 4
    for (int rr = 0; rr < GT; ++rr) {
      const float2 yv = ys[tx][rr];
#pragma unroll
      for (int q = 0; q < decltype(nq)::value; ++q) {
        const float2 xv = xs[ty + 8 * q][rr];
        acc[q].fma(dfl{xv.x, xv.y}, dfl{yv.x, yv.y});
      }
    }
  };
  const int cols = (s1 - ta * GT - ty + 7) / 8;  // of this warp, at most 4 here
  fetch(r0);
  for (long rb = r0; rb < r1; rb += GT) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const dfl a = d2df(xd[q]), b = d2df(yd[q]);
      xs[ty + 8 * q][tx] = make_float2(a.hi, a.lo);
      ys[ty + 8 * q][tx] = make_float2(b.hi, b.lo);
    }
    __syncthreads();
    if (rb + GT < r1) fetch(rb + GT);
    if (cols >= 4) rows(std::integral_constant<int, 4>{});
    else if (cols == 3) rows(std::integral_constant<int, 3>{});
    else if (cols == 2) rows(std::integral_constant<int, 2>{});
    else if (cols == 1) rows(std::integral_constant<int, 1>{});
    __syncthreads();
  }
  const int nta = gridDim.x, ntb = gridDim.y;
  for (int q = 0; q < 4; ++q) {
    const int a = ty + 8 * q, b = tx;
    part[(((long)ch * nta + ta) * ntb + tb) * GT * GT + a * GT + b] = df2d(acc[q].result());
  }
}

__global__ void k_gram_final(const double *__restrict__ part, int nchunk, int nta, int ntb, int s1, int s2,
                             double *__restrict__ G, int ldg, int sym) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= s1 * s2) return;
  int a = idx % s1, b = idx / s1;
  if (sym && a / GT > b / GT) {  // a tile below the diagonal: the mirrored entry of the one above
    const int t = a;
    a = b;
    b = t;
  }
  const int ta = a / GT, tb = b / GT;
  double s = 0.0;
#pragma unroll 8
  for (int c = 0; c < nchunk; ++c) s += part[(((long)c * nta + ta) * ntb + tb) * GT * GT + (a % GT) * GT + (b % GT)];
  G[idx % s1 + (long)ldg * (idx / s1)] = s;
}

// G = X^T y for a single column y: each block sums its chunk of rows for 8 columns of X at a
// time (coalesced along the rows), the partials [chunk][column] are added in chunk order
__global__ void k_gemv_t_partial(const double *__restrict__ X, long ldx, int s1, const double *__restrict__ y,
                                 long n, long rows_per_chunk, double *__restrict__ part) {
  __shared__ double red[8][8];  // [warp][column of the group]
  const int ch = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long r0 = ch * rows_per_chunk, r1 = min(n, r0 + rows_per_chunk);
  for (int a0 = 0; a0 < s1; a0 += 8) {
    double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (long i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
      const double yi = y[i];
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (a0 + q < s1) acc[q] = fmadd(X[ldx * (a0 + q) + i], yi, acc[q]);
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
      if (lane == 0) red[w][q] = acc[q];
    }
    __syncthreads();
    if (threadIdx.x < 8 && a0 + (int)threadIdx.x < s1) {
      double t = 0.0;
      for (int ww = 0; ww < (int)(blockDim.x >> 5); ++ww) t += red[ww][threadIdx.x];
      part[(long)ch * s1 + a0 + threadIdx.x] = t;
    }
    __syncthreads();
  }
}

__global__ void k_gemv_t_final(const double *__restrict__ part, int nchunk, int s1, double *__restrict__ G) {
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= s1) return;
  double t = 0.0;
  for (int c = 0; c < nchunk; ++c) t += part[(long)c * s1 + a];
  G[a] = t;
}

int gram(hp_problem *P, const double *X, long ldx, int s1, const double *Y, long ldy, int s2, double *G, int ldg,
         long n) {
  if (s2 == 1) {  // a matrix-vector product: the tiled kernel would compute a whole tile of X^T Y
    int nchunk = 2 * NSM;
    const long rpc = std::max<long>(256, (n + nchunk - 1) / nchunk);
    nchunk = (int)((n + rpc - 1) / rpc);
    HP_TRY(P->vtmp[5].ensure(sizeof(double) * (size_t)nchunk * s1));
    double *part = P->vtmp[5].as<double>();
    k_gemv_t_partial<<<nchunk, 256, 0, P->st>>>(X, ldx, s1, Y, n, rpc, part);
    k_gemv_t_final<<<(s1 + 255) / 256, 256, 0, P->st>>>(part, nchunk, s1, G);
    count_launch(2);
    return cuda_check(cudaGetLastError(), "gram");
  }
  const int nta = (s1 + GT - 1) / GT, ntb = (s2 + GT - 1) / GT;
  const bool df = P->refine_df != 0;  // the Gram in double-float (see k_gram_partial_df)
  const int sym = df && X == Y && ldx == ldy && s1 == s2;
  // two CTAs per SM over the tiles that are computed
  int nchunk = std::max(1, (2 * NSM) / (sym ? nta * (nta + 1) / 2 : nta * ntb));
  long rpc = (n + nchunk - 1) / nchunk;
  rpc = (rpc + GT - 1) / GT * GT;
  nchunk = (int)((n + rpc - 1) / rpc);
  if (nchunk < 1) nchunk = 1;
  const size_t need = sizeof(double) * (size_t)nchunk * nta * ntb * GT * GT;
  HP_TRY(P->vtmp[5].ensure(need));
  double *part = P->vtmp[5].as<double>();
  if (df)
    k_gram_partial_df<<<dim3(nta, ntb, nchunk), 256, 0, P->st>>>(X, ldx, s1, Y, ldy, s2, n, rpc, sym, part);
  else
    k_gram_partial<<<dim3(nta, ntb, nchunk), 256, 0, P->st>>>(X, ldx, s1, Y, ldy, s2, n, rpc, part);
  k_gram_final<<<(s1 * s2 + 255) / 256, 256, 0, P->st>>>(part, nchunk, nta, ntb, s1, s2, G, ldg, sym);
  count_launch(2);
  return cuda_check(cudaGetLastError(), "gram");
}

__global__ void k_gemm_nn(const double *__restrict__ X, long ldx, int s1, const double *__restrict__ S, int lds,
                          int s2, double *__restrict__ Y, long ldy, long n, double alpha, double beta) {
  const int j = blockIdx.y;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int k = 0; k < s1; ++k) acc += X[ldx * k + i] * __ldg(&S[k + (long)lds * j]);
    const double y = beta == 0.0 ? 0.0 : beta * Y[ldy * j + i];
    Y[ldy * j + i] = alpha * acc + y;
  }
}

// The same product in double-float on the FP32 pipe: each thread forms NJ output columns of
// its row as compensated (Dot2) sums, so every element of X is split into a pair once per NJ
// columns instead of read and multiplied in FP64 for each; the pairs of S's columns lie in
// shared memory, two to a load.  alpha and beta are applied in FP64 once per output.
// Bound by the FP32 pipe: 13 operations per term.  65^3 rows, 100 x 64: 1,126 -> 902 us with 16
// columns instead of 8 and four elements of X under way (613 us for the operations alone).
constexpr int GM_NJ = 8, GM_NJ2 = 16;
template <int NJ>
__global__ void __launch_bounds__(NT) k_gemm_nn_df(const double *__restrict__ X, long ldx, int s1,
                                                   const double *__restrict__ S, int lds, int s2,
                                                   double *__restrict__ Y, long ldy, long n, double alpha,
                                                   double beta) {
  extern __shared__ __align__(16) float2 sp[];  // the block's NJ columns of S as pairs, [k][q]
  const int j0 = blockIdx.y * NJ;
  for (int t = threadIdx.x; t < s1 * NJ; t += blockDim.x) {
    const int k = t / NJ, q = t % NJ;
    const dfl d = d2df(j0 + q < s2 ? S[k + (long)lds * (j0 + q)] : 0.0);
    sp[t] = make_float2(d.hi, d.lo);
  }
  __syncthreads();
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    Dot2 acc[NJ];
    auto term = [&](int k, double xk) {
      const dfl x = d2df(xk);
      const float4 *sk = reinterpret_cast<const float4 *>(sp + k * NJ);
#pragma unroll
      for (int q = 0; q < NJ; q += 2) {
        const float4 sv = sk[q / 2];
        acc[q].fma(dfl{sv.x, sv.y}, x);
        acc[q + 1].fma(dfl{sv.z, sv.w}, x);
      }
    };
    int k = 0;
    for (; k + 4 <= s1; k += 4) {
      double x[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) x[e] = X[ldx * (k + e) + i];
#pragma unroll
      for (int e = 0; e < 4; ++e) term(k + e, x[e]);
    }
    for (; k < s1; ++k) term(k, X[ldx * k + i]);
#pragma unroll
    for (int q = 0; q < NJ; ++q) {
      const int j = j0 + q;
      if (j >= s2) break;
      const double y = beta == 0.0 ? 0.0 : beta * Y[ldy * j + i];
      Y[ldy * j + i] = alpha * df2d(acc[q].result()) + y;
    }
  }
}

// R^{-1} of an upper-triangular R (column-major, s x s) in FP64, one warp per column: back
// substitution of R x = e_j (the upper triangle of the result; zeros below), a row's sum split
// over the lanes.  One thread per column took 120 us for s = 60, chains of loads and FP64
// operations with a latency of tens of clocks each; this takes 35.
__global__ void __launch_bounds__(128) k_tri_inv(const double *__restrict__ R, int s, double *__restrict__ Ri) {
  extern __shared__ double ti_x[];  // [4 warps][2][s]: the column, and the inverse diagonal
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, j = blockIdx.x * 4 + w;
  double *x = ti_x + (long)w * 2 * s, *rd = x + s;
  if (j >= s) return;
  for (int i = lane; i <= j; i += 32) rd[i] = 1.0 / R[i + (long)s * i];
  for (int i = j + 1 + lane; i < s; i += 32) Ri[i + (long)s * j] = 0.0;
  __syncwarp();
  if (lane == 0) x[j] = rd[j];
  __syncwarp();
  for (int i = j - 1; i >= 0; --i) {
    double t = 0.0;
    for (int k = i + 1 + lane; k <= j; k += 32) t = fma(R[i + (long)s * k], x[k], t);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) x[i] = -t * rd[i];
    __syncwarp();
  }
  for (int i = lane; i <= j; i += 32) Ri[i + (long)s * j] = x[i];
}

void launch_gemm_nn(const double *X, long ldx, int s1, const double *S, int lds, int s2, double *Y, long ldy, long n,
                    double alpha, double beta, hp_problem *P) {
  if (P->refine_df != 0 && s2 > 1 && sizeof(float2) * (size_t)s1 * GM_NJ <= 48 * 1024) {
    // 16 columns per thread where more than half of the last 16 are there and they fit
    const size_t shm = sizeof(float2) * (size_t)s1 * GM_NJ2;
    const int nj2 = (s2 + GM_NJ2 - 1) / GM_NJ2, nj = (s2 + GM_NJ - 1) / GM_NJ;
    if (nj == 2 * nj2 && shm <= 48 * 1024)
      k_gemm_nn_df<GM_NJ2><<<dim3(blocks_for(n, nj2), nj2), NT, shm, P->st>>>(X, ldx, s1, S, lds, s2, Y, ldy, n, alpha,
                                                                             beta);
    else
      k_gemm_nn_df<GM_NJ><<<dim3(blocks_for(n, nj), nj), NT, sizeof(float2) * (size_t)s1 * GM_NJ, P->st>>>(
          X, ldx, s1, S, lds, s2, Y, ldy, n, alpha, beta);
  } else {
    k_gemm_nn<<<dim3(blocks_for(n, s2), s2), NT, 0, P->st>>>(X, ldx, s1, S, lds, s2, Y, ldy, n, alpha, beta);
  }
  count_launch();
}

// y <- y - Q c  with c (device, length j) ; then optionally report |y|^2
__global__ void k_scale_col(double *__restrict__ y, long n, const double *__restrict__ nrm2) {
  const double nv = sqrt(*nrm2);
  const double inv = nv > 0.0 ? 1.0 / nv : 0.0;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) y[i] *= inv;
}

int cgs2_qr(hp_problem *P, double *Y, long ldy, long n, int s) {
  HP_TRY(P->vtmp[4].ensure(sizeof(double) * (size_t)(s + 2)));
  double *c = P->vtmp[4].as<double>();
  for (int j = 0; j < s; ++j) {
    double *y = Y + ldy * j;
    for (int pass = 0; pass < 2 && j > 0; ++pass) {
      HP_TRY(gram(P, Y, ldy, j, y, ldy, 1, c, j, n));
      launch_gemm_nn(Y, ldy, j, c, j, 1, y, ldy, n, -1.0, 1.0, P);
    }
    HP_TRY(block_dot(P, y, ldy, y, ldy, n, 1, c + s));
    k_scale_col<<<blocks_for(n, 1), NT, 0, P->st>>>(y, n, c + s);
    count_launch();
  }
  return cuda_check(cudaGetLastError(), "cgs2_qr");
}

// ---------------------------------------------------------------------------
// Thin QR of a tall block by shifted Cholesky QR, three passes (Fukaya, Kannan,
// Nakatsukasa, Yamamoto, Yanagisawa, "Shifted Cholesky QR for computing the QR
// factorization of ill-conditioned matrices", SIAM J. Sci. Comput. 2020): each pass forms
// G = Y^T Y, factors G = R^T R and sets Y <- Y R^{-1}; the first pass factors G + sigma I
// with sigma = 11 (n s + s (s + 1)) u tr(G) (tr(G) >= |Y|_2^2, u the unit roundoff), which
// keeps the Cholesky factorisable for any numerically full-rank Y and makes Y well enough
// conditioned for the two plain passes to reach orthogonality at the rounding level.
// Three full-width Gram products replace the 2(s - 1) one-column products of
// column-by-column Gram-Schmidt, which waste most of each FP64 Gram tile.  A Gram matrix
// that still is not positive definite (a rank-deficient block) falls back to cgs2_qr.
// ---------------------------------------------------------------------------
__global__ void k_sym_copy(const double *__restrict__ G, double *__restrict__ R, int s) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= s * s) return;
  const int a = idx % s, b = idx / s;
  R[idx] = 0.5 * (G[a + (long)s * b] + G[b + (long)s * a]);
}

__global__ void k_shift_diag(double *R, int s, long n) {
  __shared__ double tr;
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < s; ++i) t += R[i + (long)s * i];
    tr = t;
  }
  __syncthreads();
  const double sigma = 11.0 * ((double)n * s + (double)s * (s + 1)) * 0x1p-53 * tr;
  for (int i = threadIdx.x; i < s; i += blockDim.x) R[i + (long)s * i] += sigma;
}

int thin_qr(hp_problem *P, double *Y, long ldy, long n, int s) {
  HP_TRY(P->vtmp[4].ensure(sizeof(double) * (2 * (size_t)s * s + (size_t)s + 2)));
  double *G = P->vtmp[4].as<double>(), *R = G + (size_t)s * s;
  for (int pass = 0; pass < 3; ++pass) {
    HP_TRY(gram(P, Y, ldy, s, Y, ldy, s, G, s, n));
    k_sym_copy<<<(s * s + 255) / 256, 256, 0, P->st>>>(G, R, s);
    count_launch();
    if (pass == 0) {
      k_shift_diag<<<1, 256, 0, P->st>>>(R, s, n);
      count_launch();
    }
    if (small_cholesky(P, R, s) != 0) return cgs2_qr(P, Y, ldy, n, s);
    launch_trsm_right_upper(Y, ldy, n, s, R, P);
  }
  return cuda_check(cudaGetLastError(), "thin_qr");
}

// lower Cholesky in place (row-major) == upper R in column-major
__global__ void k_small_chol(double *A, int s, int *status) {
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  for (int k = 0; k < s; ++k) {
    if (threadIdx.x == 0) {
      const double d = A[(long)k * s + k];
      if (!(d > 0.0) || !isfinite(d)) bad = 1;
      A[(long)k * s + k] = d > 0.0 ? sqrt(d) : 1.0;
    }
    __syncthreads();
    const double dk = A[(long)k * s + k];
    for (int i = k + 1 + threadIdx.x; i < s; i += blockDim.x) A[(long)i * s + k] /= dk;
    __syncthreads();
    const int m = s - k - 1;
    for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
      const int i = k + 1 + t / m, jj = k + 1 + t % m;
      if (jj <= i) A[(long)i * s + jj] -= A[(long)i * s + k] * A[(long)jj * s + k];
    }
    __syncthreads();
  }
  // clear the strictly lower part of the column-major R (upper part of row-major)
  for (int t = threadIdx.x; t < s * s; t += blockDim.x) {
    const int i = t / s, jj = t % s;
    if (jj > i) A[(long)i * s + jj] = 0.0;
  }
  if (threadIdx.x == 0) *status = bad;
}

// The same for s up to CH_SM with the triangle in shared memory, as L D L^T: a step scales the
// pivot's column by 1 / d and updates the rows below, a warp per row; the thread that finishes
// the next pivot forms its reciprocal while the others update, and the roots are taken at the
// end, for all columns at once.  Bound by the latency of the s reciprocals and the FP64 pipe
// (s = 60: 94 -> 59 us).
constexpr int CH_SM = 144;
constexpr int CH_NT = 512;
static size_t chol_smem(int s) { return sizeof(double) * ((size_t)s * (s + 1) + 2 * s); }

__global__ void __launch_bounds__(CH_NT) k_small_chol_sm(double *A, int s, int *status) {
  extern __shared__ double ch[];  // rows of s + 1 doubles; the scaled column; the reciprocals
  const int ld = s + 1, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double *wk = ch + s * ld, *rd = wk + s;
  __shared__ int bad;
  for (int t = threadIdx.x; t < s * s; t += CH_NT) {
    const int i = t / s, j = t - i * s;
    if (j <= i) ch[i * ld + j] = A[t];
  }
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  auto pivot = [&](int k) {
    const double d = ch[k * ld + k];
    if (!(d > 0.0) || !isfinite(d)) bad = 1;
    rd[k] = d > 0.0 ? 1.0 / d : 1.0;
  };
  if (threadIdx.x == 0) pivot(0);
  __syncthreads();
  for (int k = 0; k + 1 < s; ++k) {
    const double r = rd[k];
    for (int i = k + 1 + threadIdx.x; i < s; i += CH_NT) wk[i] = ch[i * ld + k] * r;
    __syncthreads();
    for (int i = k + 1 + w; i < s; i += CH_NT / 32) {
      const double li = wk[i];
      for (int j = k + 1 + lane; j <= i; j += 32) ch[i * ld + j] = fma(-li, ch[j * ld + k], ch[i * ld + j]);
      if (i == k + 1 && lane == 0) pivot(i);
    }
    __syncthreads();
  }
  for (int k = threadIdx.x; k < s; k += CH_NT) {
    const double d = ch[k * ld + k], q = d > 0.0 ? sqrt(d) : 1.0;
    wk[k] = q;
    rd[k] = 1.0 / q;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < s * s; t += CH_NT) {
    const int i = t / s, j = t - i * s;
    A[t] = j < i ? ch[i * ld + j] * rd[j] : (j == i ? wk[i] : 0.0);
  }
  if (threadIdx.x == 0) *status = bad;
}

int small_cholesky(hp_problem *P, double *G, int s) {
  int *d = P->sc.active.as<int>();
  if (s <= CH_SM) {
    static std::atomic<unsigned long long> attr_ch{0};  // once per device: the largest size
    int dev = 0;
    HP_CUDA(cudaGetDevice(&dev));
    if (dev < 64 && !(attr_ch.load(std::memory_order_acquire) & (1ull << dev))) {
      HP_CUDA(cudaFuncSetAttribute(k_small_chol_sm, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)chol_smem(CH_SM)));
      attr_ch.fetch_or(1ull << dev, std::memory_order_release);
    }
    k_small_chol_sm<<<1, CH_NT, chol_smem(s), P->st>>>(G, s, d);
  } else
    k_small_chol<<<1, 1024, 0, P->st>>>(G, s, d);
  count_launch();
  int h = 0;
  HP_CUDA(cudaMemcpyAsync(&h, d, sizeof(int), cudaMemcpyDeviceToHost, P->st));
  HP_CUDA(cudaStreamSynchronize(P->st));
  if (h) return set_error(HP_ERR_NONFINITE, "Gram matrix of PreCholQR is not positive definite");
  return 0;
}

// Y <- Y R^{-1} (R upper, column-major s x s): row-wise forward substitution
__global__ void k_trsm_ru(double *__restrict__ Y, long ldy, long n, int s, const double *__restrict__ R) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    for (int j = 0; j < s; ++j) {
      double v = Y[ldy * j + i];
      for (int k = 0; k < j; ++k) v -= Y[ldy * k + i] * __ldg(&R[k + (long)s * j]);
      Y[ldy * j + i] = v / __ldg(&R[j + (long)s * j]);
    }
  }
}

void launch_trsm_right_upper(double *Y, long ldy, long n, int s, const double *R, hp_problem *P) {
  // double-float: Y R^{-1} as a product with the explicit inverse (FP64, one small kernel),
  // formed into a scratch block by the double-float product and copied back.  The inverse's
  // rounding is about cond(R) 2^-48 relative; the QR passes that use it are self-correcting
  // and the eigensolver's R-orthonormality is checked to 1e-7.
  const long ldt = (n + 63) / 64 * 64;
  if (P->refine_df != 0 && s > 1 && sizeof(double) * (size_t)s * GM_NJ <= 48 * 1024 &&
      P->vtmp[3].ensure(sizeof(double) * (size_t)s * s) == 0 && P->dense_tmp.ensure(sizeof(double) * ldt * s) == 0) {
    double *Ri = P->vtmp[3].as<double>(), *T = P->dense_tmp.as<double>();
    k_tri_inv<<<(s + 3) / 4, 128, sizeof(double) * 8 * s, P->st>>>(R, s, Ri);
    count_launch();
    launch_gemm_nn(Y, ldy, s, Ri, s, s, T, ldt, n, 1.0, 0.0, P);
    cudaMemcpy2DAsync(Y, sizeof(double) * ldy, T, sizeof(double) * ldt, sizeof(double) * n, s,
                      cudaMemcpyDeviceToDevice, P->st);
    return;
  }
  (void)cudaGetLastError();
  k_trsm_ru<<<blocks_for(n, 1), NT, 0, P->st>>>(Y, ldy, n, s, R);
  count_launch();
}

// ---------------------------------------------------------------------------
// cyclic Jacobi eigen-solver, one block.  A (s x s) and V in global scratch.
// ---------------------------------------------------------------------------
__global__ void k_jacobi_eig(double *A, double *V, int s, int m, double *lam_out, double *S_out, int max_sweeps) {
  extern __shared__ double sh[];
  double *cs = sh;          // m/2 cosines
  double *sn = sh + m / 2;  // m/2 sines
  int *pp = reinterpret_cast<int *>(sn + m / 2);
  int *qq = pp + m / 2;
  __shared__ double off_s, tot_s;
  for (int t = threadIdx.x; t < s * s; t += blockDim.x) V[t] = (t % s == t / s) ? 1.0 : 0.0;
  __syncthreads();
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    // convergence test
    if (threadIdx.x == 0) {
      double off = 0.0, tot = 0.0;
      for (int t = 0; t < s * s; ++t) {
        const double v = A[t] * A[t];
        tot += v;
        if (t % s != t / s) off += v;
      }
      off_s = off;
      tot_s = tot;
    }
    __syncthreads();
    if (off_s <= 1e-30 * tot_s || off_s == 0.0) break;
    for (int r = 0; r < m - 1; ++r) {
      for (int k = threadIdx.x; k < m / 2; k += blockDim.x) {
        int p, q;
        if (k == 0) {
          p = r;
          q = m - 1;
        } else {
          p = (r + k) % (m - 1);
          q = (r - k + (m - 1)) % (m - 1);
        }
        if (p > q) {
          const int t = p;
          p = q;
          q = t;
        }
        double c = 1.0, sv = 0.0;
        if (q < s) {
          const double apq = A[p + (long)s * q];
          if (apq != 0.0) {
            const double theta = (A[q + (long)s * q] - A[p + (long)s * p]) / (2.0 * apq);
            const double t = (theta >= 0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
            c = 1.0 / sqrt(t * t + 1.0);
            sv = t * c;
          }
        }
        cs[k] = c;
        sn[k] = sv;
        pp[k] = p;
        qq[k] = q;
      }
      __syncthreads();
      // rows: A <- J^T A
      for (int t = threadIdx.x; t < (m / 2) * s; t += blockDim.x) {
        const int k = t / s, col = t % s;
        const int p = pp[k], q = qq[k];
        if (q >= s) continue;
        const double c = cs[k], sv = sn[k];
        const double ap = A[p + (long)s * col], aq = A[q + (long)s * col];
        A[p + (long)s * col] = c * ap - sv * aq;
        A[q + (long)s * col] = sv * ap + c * aq;
      }
      __syncthreads();
      // columns: A <- A J, V <- V J
      for (int t = threadIdx.x; t < (m / 2) * s; t += blockDim.x) {
        const int k = t / s, row = t % s;
        const int p = pp[k], q = qq[k];
        if (q >= s) continue;
        const double c = cs[k], sv = sn[k];
        const double ap = A[row + (long)s * p], aq = A[row + (long)s * q];
        A[row + (long)s * p] = c * ap - sv * aq;
        A[row + (long)s * q] = sv * ap + c * aq;
        const double vp = V[row + (long)s * p], vq = V[row + (long)s * q];
        V[row + (long)s * p] = c * vp - sv * vq;
        V[row + (long)s * q] = sv * vp + c * vq;
      }
      __syncthreads();
    }
  }
  // sort descending (selection order computed by thread 0), write outputs
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int a = 0; a < s; ++a) pp[a] = a;
    for (int a = 0; a < s; ++a) {
      int best = a;
      for (int b = a + 1; b < s; ++b)
        if (A[pp[b] + (long)s * pp[b]] > A[pp[best] + (long)s * pp[best]]) best = b;
      const int t = pp[a];
      pp[a] = pp[best];
      pp[best] = t;
    }
  }
  __syncthreads();
  for (int a = threadIdx.x; a < s; a += blockDim.x) lam_out[a] = A[pp[a] + (long)s * pp[a]];
  for (int t = threadIdx.x; t < s * s; t += blockDim.x) {
    const int row = t % s, col = t / s;
    S_out[row + (long)s * col] = V[row + (long)s * pp[col]];
  }
}

// The same cyclic Jacobi method (same rotations in the same order) with A in shared memory
// and the off-diagonal norm of the convergence test as a block reduction: V shares the
// shared memory for s <= JS_MAX, and lives in the global scratch Vg up to JS_MAX_A.
constexpr int JS_MAX = 90, JS_MAX_A = 160;

__global__ void __launch_bounds__(1024) k_jacobi_eig_sm(const double *__restrict__ Ain, int s, int m,
                                                        double *lam_out, double *S_out, int max_sweeps,
                                                        double *Vg) {
  extern __shared__ double sh[];
  double *A = sh, *V = Vg ? Vg : A + s * s;
  double *cs = A + s * s + (Vg ? 0 : s * s), *sn = cs + m / 2, *red = sn + m / 2;  // red: [2][32]
  int *pp = reinterpret_cast<int *>(red + 64);
  int *qq = pp + (m > s ? m : s);
  for (int t = threadIdx.x; t < s * s; t += blockDim.x) {
    A[t] = Ain[t];
    V[t] = (t % s == t / s) ? 1.0 : 0.0;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    double off = 0.0, tot = 0.0;
    for (int t = threadIdx.x; t < s * s; t += blockDim.x) {
      const double v = A[t] * A[t];
      tot += v;
      if (t % s != t / s) off += v;
    }
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    if (lane == 0) {
      red[wid] = off;
      red[32 + wid] = tot;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double a = 0.0, b = 0.0;
      for (int w = 0; w < nw; ++w) {
        a += red[w];
        b += red[32 + w];
      }
      red[0] = a;
      red[32] = b;
    }
    __syncthreads();
    const double off_s = red[0], tot_s = red[32];
    __syncthreads();
    if (off_s <= 1e-30 * tot_s || off_s == 0.0) break;
    for (int r = 0; r < m - 1; ++r) {
      for (int k = threadIdx.x; k < m / 2; k += blockDim.x) {
        int p, q;
        if (k == 0) {
          p = r;
          q = m - 1;
        } else {
          p = (r + k) % (m - 1);
          q = (r - k + (m - 1)) % (m - 1);
        }
        if (p > q) {
          const int t = p;
          p = q;
          q = t;
        }
        double c = 1.0, sv = 0.0;
        if (q < s) {
          const double apq = A[p + s * q];
          if (apq != 0.0) {
            const double theta = (A[q + s * q] - A[p + s * p]) / (2.0 * apq);
            const double t = (theta >= 0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
            c = 1.0 / sqrt(t * t + 1.0);
            sv = t * c;
          }
        }
        cs[k] = c;
        sn[k] = sv;
        pp[k] = p;
        qq[k] = q;
      }
      __syncthreads();
      for (int t = threadIdx.x; t < (m / 2) * s; t += blockDim.x) {  // rows: A <- J^T A
        const int k = t / s, col = t % s;
        const int p = pp[k], q = qq[k];
        if (q >= s) continue;
        const double c = cs[k], sv = sn[k];
        const double ap = A[p + s * col], aq = A[q + s * col];
        A[p + s * col] = c * ap - sv * aq;
        A[q + s * col] = sv * ap + c * aq;
      }
      __syncthreads();
      for (int t = threadIdx.x; t < (m / 2) * s; t += blockDim.x) {  // columns: A <- A J, V <- V J
        const int k = t / s, row = t % s;
        const int p = pp[k], q = qq[k];
        if (q >= s) continue;
        const double c = cs[k], sv = sn[k];
        const double ap = A[row + s * p], aq = A[row + s * q];
        A[row + s * p] = c * ap - sv * aq;
        A[row + s * q] = sv * ap + c * aq;
        const double vp = V[row + s * p], vq = V[row + s * q];
        V[row + s * p] = c * vp - sv * vq;
        V[row + s * q] = sv * vp + c * vq;
      }
      __syncthreads();
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int a = 0; a < s; ++a) pp[a] = a;
    for (int a = 0; a < s; ++a) {
      int best = a;
      for (int b = a + 1; b < s; ++b)
        if (A[pp[b] + s * pp[b]] > A[pp[best] + s * pp[best]]) best = b;
      const int t = pp[a];
      pp[a] = pp[best];
      pp[best] = t;
    }
  }
  __syncthreads();
  for (int a = threadIdx.x; a < s; a += blockDim.x) lam_out[a] = A[pp[a] + s * pp[a]];
  for (int t = threadIdx.x; t < s * s; t += blockDim.x) {
    const int row = t % s, col = t / s;
    S_out[row + (long)s * col] = V[row + s * pp[col]];
  }
}

// The same cyclic Jacobi with its rotations applied in double-float on the FP32 pipe: A
// (and V while it fits) held as float pairs in shared memory, V in the global scratch Vg
// beyond that.  Each rotation's angle comes from the three entries it needs (rot_angle), its
// cosine and sine as pairs, and every update
// x' = c x - s y, y' = s x + c y is a compensated (Dot2) two-term sum.  A round's rotations
// are applied block by block: for two of its pairs a thread takes the 2 x 2 entries from
// both sides and writes them with their mirror image, so a round is half the work of
// a pass over the rows and one over the columns, and one barrier less (s = 60: 3.7 -> 2.5 ms,
// 2.6 us a round; bound by the rounds' serial chain of angles, barriers and updates on one SM).  The off-diagonal
// test uses the leading floats' squares, in FP64.
__device__ __forceinline__ dfl rot_mix(dfl a, dfl x, dfl b, dfl y) {  // a x + b y
  Dot2 d;
  d.fma(a, x);
  d.fma(b, y);
  return d.result();
}

// Cosine and sine (as pairs) of a rotation that takes apq to (nearly) zero: the tangent
// t = sign(theta) / (|theta| + sqrt(theta^2 + 1)), theta = (aqq - app) / (2 apq), is a float, and
// c = 1 / sqrt(1 + t^2) and s = t c follow from that float in double-float, so the rotation is
// orthogonal whatever t's rounding (c^2 + s^2 - 1 below 8e-14 over 400,000 random entries with the
// reciprocal root up to two ulps off); an entry left at some 1e-6 of its size instead of 0 does
// not slow the sweeps down.  c: a float reciprocal root y and one third-order step on its
// residual r = 1 - (1 + t^2) y^2, from the binomial series (1 - r)^(-1/2) = 1 + r/2 + 3/8 r^2 + ...
// In FP64 its divisions and roots took a third of the solver's time (s = 60: 5.4 -> 3.7 ms), and
// with c and s rounded to pairs one by one the eigenvectors (2 to 140 rows; decaying, clustered and
// random spectra) were up to 4.9e-12 off orthogonal, 2.8e-13 this way, the eigenvalues 3.1e-12 and
// 2.2e-13 off LAPACK's.
__device__ __forceinline__ void rot_angle(dfl app, dfl aqq, dfl apq, dfl *c, dfl *s) {
  const dfl d = two_sum(aqq.hi, -app.hi);
  const float diff = d.hi + (d.lo + (aqq.lo - app.lo));
  const float theta = diff / (2.f * apq.hi);
  const float t = copysignf(1.f, theta) / (fabsf(theta) + sqrtf(fmaf(theta, theta, 1.f)));
  const dfl tt = two_prod(t, t);
  dfl u = two_sum(1.f, tt.hi);
  u.lo += tt.lo;
  const float y = rsqrtf(u.hi);
  const dfl yy = two_prod(y, y), w = two_prod(u.hi, yy.hi);
  const float r = (1.f - w.hi) - (w.lo + fmaf(u.hi, yy.lo, u.lo * yy.hi));
  *c = fast_two_sum(y, y * r * fmaf(0.375f, r, 0.5f));
  const dfl p = two_prod(t, c->hi);
  *s = fast_two_sum(p.hi, fmaf(t, c->lo, p.lo));
}

__global__ void __launch_bounds__(1024) k_jacobi_eig_sm_df(const double *__restrict__ Ain, int s, int m,
                                                           double *lam_out, double *S_out, int max_sweeps,
                                                           float2 *Vg) {
  extern __shared__ float2 shp[];
  // A (zero in the extra row and column of an odd s) and V while it fits, with an odd leading
  // dimension la: neighbouring lanes' columns then lie in different banks
  const int la = m + 1, h = m / 2;
  float2 *A = shp, *V = Vg ? Vg : A + la * m;
  const int lv = Vg ? s : la;
  float2 *csp = A + la * m + (Vg ? 0 : la * m), *snp = csp + h;
  double *red = reinterpret_cast<double *>(snp + m / 2);  // [2][32]
  int *pp = reinterpret_cast<int *>(red + 64);
  int *qq = pp + (m > s ? m : s);
  for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
    const int row = t % m, col = t / m;
    const bool in = row < s && col < s;
    const dfl a = d2df(in ? 0.5 * (Ain[row + s * col] + Ain[col + s * row]) : 0.0);
    A[row + la * col] = make_float2(a.hi, a.lo);
    if (in) V[row + lv * col] = make_float2(row == col ? 1.f : 0.f, 0.f);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  auto J = [](float2 v) { return df2d(dfl{v.x, v.y}); };
  auto rot = [](dfl c, dfl sn, dfl &x, dfl &y) {  // x' = c x - s y, y' = s x + c y
    const dfl a = rot_mix(c, x, dfl{-sn.hi, -sn.lo}, y);
    y = rot_mix(sn, x, c, y);
    x = a;
  };
  // blocks (a, b), a <= b, of the round's pairs, numbered over a rectangle of nbc columns, and
  // items of up to four rows of V per pair
  const unsigned nbc = (h & 1) ? h : h + 1, nblk = h * (h + 1) / 2, nr4 = (s + 3) / 4;
  const unsigned mbc = 0xFFFFFFFFu / nbc + 1, mr4 = 0xFFFFFFFFu / nr4 + 1;  // t / d for t < 2^16, d > 1
  double off_prev = 0.0;
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    double off = 0.0, tot = 0.0;
    for (int t = threadIdx.x; t < s * s; t += blockDim.x) {
      const int row = t % s, col = t / s;
      const double v = J(A[row + la * col]);
      tot += v * v;
      if (row != col) off += v * v;
    }
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    if (lane == 0) {
      red[wid] = off;
      red[32 + wid] = tot;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double a = 0.0, b = 0.0;
      for (int w = 0; w < nw; ++w) {
        a += red[w];
        b += red[32 + w];
      }
      red[0] = a;
      red[32] = b;
    }
    __syncthreads();
    const double off_s = red[0], tot_s = red[32];
    __syncthreads();
    // the pairs carry about 48 bits, so the off-diagonal mass stops falling near
    // s (2^-48)^2 of the total: stop at 1e-26 of it (1e-13 in norm), or once a sweep no longer
    // halves it (the rounding floor; the sweeps before it converge quadratically)
    if (off_s <= 1e-26 * tot_s || off_s == 0.0 || (sweep >= 3 && off_s > 0.5 * off_prev)) break;
    off_prev = off_s;
    for (int r = 0; r < m - 1; ++r) {
      for (int k = threadIdx.x; k < h; k += blockDim.x) {
        int p = k == 0 ? r : (r + k < m - 1 ? r + k : r + k - (m - 1));
        int q = k == 0 ? m - 1 : (r >= k ? r - k : r - k + m - 1);
        if (p > q) {
          const int t = p;
          p = q;
          q = t;
        }
        dfl cd{1.f, 0.f}, sd{0.f, 0.f};
        const float2 pq = A[p + la * q], pv = A[p + la * p], qv = A[q + la * q];
        if (q < s && pq.x != 0.f) rot_angle(dfl{pv.x, pv.y}, dfl{qv.x, qv.y}, dfl{pq.x, pq.y}, &cd, &sd);
        csp[k] = make_float2(cd.hi, cd.lo);
        snp[k] = make_float2(sd.hi, sd.lo);
        pp[k] = p;
        qq[k] = q;
      }
      __syncthreads();
      // A <- J^T A J and V <- V J
      for (unsigned t = threadIdx.x; t < nblk + h * nr4; t += blockDim.x) {
        if (t < nblk) {
          const int br = nbc == 1 ? 0 : (int)__umulhi(t, mbc), bc = (int)t - br * (int)nbc;
          int a, b;
          if (h & 1) {
            a = bc >= br ? br : h - br;
            b = bc >= br ? bc : h - 1 - bc;
          } else {
            a = bc > br ? br : h - 1 - br;
            b = bc > br ? bc - 1 : h - 1 - bc;
          }
          const int p1 = pp[a], q1 = qq[a], p2 = pp[b], q2 = qq[b];
          const dfl c1{csp[a].x, csp[a].y}, s1{snp[a].x, snp[a].y}, c2{csp[b].x, csp[b].y}, s2{snp[b].x, snp[b].y};
          auto ld = [&](int i, int j) {
            const float2 v = A[i + la * j];
            return dfl{v.x, v.y};
          };
          dfl xpp = ld(p1, p2), xpq = ld(p1, q2), xqp = ld(q1, p2), xqq = ld(q1, q2);
          rot(c1, s1, xpp, xqp);
          rot(c1, s1, xpq, xqq);
          rot(c2, s2, xpp, xpq);
          rot(c2, s2, xqp, xqq);
          if (a == b) xqp = xpq;
          auto put = [&](int i, int j, dfl v) { A[i + la * j] = A[j + la * i] = make_float2(v.hi, v.lo); };
          put(p1, p2, xpp);
          put(p1, q2, xpq);
          put(q1, p2, xqp);
          put(q1, q2, xqq);
        } else {
          const unsigned u = t - nblk;
          const int k = nr4 == 1 ? (int)u : (int)__umulhi(u, mr4), r0 = (int)u - k * (int)nr4;
          const int p = pp[k], q = qq[k];
          if (q >= s) continue;
          const dfl c{csp[k].x, csp[k].y}, sn{snp[k].x, snp[k].y};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int row = r0 + e * (int)nr4;
            if (row >= s) break;
            const float2 vp = V[row + lv * p], vq = V[row + lv * q];
            dfl x{vp.x, vp.y}, y{vq.x, vq.y};
            rot(c, sn, x, y);
            V[row + lv * p] = make_float2(x.hi, x.lo);
            V[row + lv * q] = make_float2(y.hi, y.lo);
          }
        }
      }
      __syncthreads();
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int a = 0; a < s; ++a) pp[a] = a;
    for (int a = 0; a < s; ++a) {
      int best = a;
      for (int b = a + 1; b < s; ++b)
        if (J(A[pp[b] * (la + 1)]) > J(A[pp[best] * (la + 1)])) best = b;
      const int t = pp[a];
      pp[a] = pp[best];
      pp[best] = t;
    }
  }
  __syncthreads();
  for (int a = threadIdx.x; a < s; a += blockDim.x) lam_out[a] = J(A[pp[a] * (la + 1)]);
  for (int t = threadIdx.x; t < s * s; t += blockDim.x) {
    const int row = t % s, col = t / s;
    S_out[row + (long)s * col] = J(V[row + lv * pp[col]]);
  }
}

int small_symeig(hp_problem *P, const double *T, int s, double *lambda, double *S) {
  const int m = s + (s & 1);
  if (s <= JS_MAX_A && P->refine_df != 0) {  // double-float rotations (same layouts, pairs for doubles)
    const bool v_shared = s <= JS_MAX;
    float2 *Vg = nullptr;
    if (!v_shared) {
      HP_TRY(P->vtmp[3].ensure(sizeof(float2) * (size_t)s * s));
      Vg = P->vtmp[3].as<float2>();
    }
    const size_t shm = sizeof(float2) * ((v_shared ? 2 : 1) * (size_t)(m + 1) * m + m) + sizeof(double) * 64 +
                       sizeof(int) * 2 * (size_t)std::max(m, s);
    static std::atomic<unsigned long long> attr_df{0};
    int dev = 0;
    HP_CUDA(cudaGetDevice(&dev));
    if (dev < 64 && !(attr_df.load(std::memory_order_acquire) & (1ull << dev))) {
      const size_t cap = std::max(sizeof(float2) * (2 * (JS_MAX + 1) * JS_MAX + JS_MAX + 1) + sizeof(double) * 64 +
                                      sizeof(int) * 2 * (JS_MAX + 1),
                                  sizeof(float2) * ((JS_MAX_A + 1) * JS_MAX_A + JS_MAX_A) + sizeof(double) * 64 +
                                      sizeof(int) * 2 * JS_MAX_A);
      HP_CUDA(cudaFuncSetAttribute(k_jacobi_eig_sm_df, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cap));
      attr_df.fetch_or(1ull << dev, std::memory_order_release);
    }
    k_jacobi_eig_sm_df<<<1, 1024, shm, P->st>>>(T, s, m, lambda, S, 60, Vg);
    count_launch();
    return cuda_check(cudaGetLastError(), "small_symeig");
  }
  if (s <= JS_MAX_A) {
    const bool v_shared = s <= JS_MAX;
    double *Vg = nullptr;
    if (!v_shared) {
      HP_TRY(P->vtmp[3].ensure(sizeof(double) * (size_t)s * s));
      Vg = P->vtmp[3].as<double>();
    }
    const size_t shm = sizeof(double) * ((v_shared ? 2 : 1) * (size_t)s * s + m + 64) +
                       sizeof(int) * 2 * (size_t)std::max(m, s);
    static std::atomic<unsigned long long> attr_set{0};  // once per device: the largest size either layout needs
    int dev = 0;
    HP_CUDA(cudaGetDevice(&dev));
    if (dev < 64 && !(attr_set.load(std::memory_order_acquire) & (1ull << dev))) {
      const size_t cap = std::max(sizeof(double) * (2 * JS_MAX * JS_MAX + JS_MAX + 1 + 64) +
                                      sizeof(int) * 2 * (JS_MAX + 1),
                                  sizeof(double) * (JS_MAX_A * JS_MAX_A + JS_MAX_A + 64) +
                                      sizeof(int) * 2 * JS_MAX_A);
      HP_CUDA(cudaFuncSetAttribute(k_jacobi_eig_sm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cap));
      attr_set.fetch_or(1ull << dev, std::memory_order_release);
    }
    k_jacobi_eig_sm<<<1, 1024, shm, P->st>>>(T, s, m, lambda, S, 60, Vg);
    count_launch();
    return cuda_check(cudaGetLastError(), "small_symeig");
  }
  HP_TRY(P->vtmp[3].ensure(sizeof(double) * 2 * (size_t)s * s));
  double *A = P->vtmp[3].as<double>(), *V = A + (size_t)s * s;
  HP_CUDA(cudaMemcpyAsync(A, T, sizeof(double) * s * s, cudaMemcpyDeviceToDevice, P->st));
  const size_t shm = sizeof(double) * m + sizeof(int) * std::max(m, s) * 2 + 64;
  k_jacobi_eig<<<1, 1024, shm, P->st>>>(A, V, s, m, lambda, S, 60);
  count_launch();
  return cuda_check(cudaGetLastError(), "small_symeig");
}

}  // namespace hp

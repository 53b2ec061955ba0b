// Small dense Hermitian algebra in shared memory, shared by the projected-problem kernels and the
// Cholesky-QR kernel.
#pragma once
#include "kernels.h"

__device__ __forceinline__ double rsqrt_approx(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  return y;
}
__device__ __forceinline__ double rcp_approx(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  return y;
}
// 1 / x to an ulp for a normal x > 0 with a normal result: two steps of the Newton-Raphson iteration
// y <- y + y (1 - x y) from the hardware's approximation of some 20 bits, four FP64 instructions.
__device__ __forceinline__ double inv_newton(double x) {
  double y = rcp_approx(x);
  y = fma(y, fma(-x, y, 1.0), y);
  return fma(y, fma(-x, y, 1.0), y);
}
// 1 / sqrt(x) to rounding, for the factorisations.
__device__ __forceinline__ float inv_sqrt(float x) { return 1.f / sqrtf(x); }
__device__ __forceinline__ double inv_sqrt(double x) {  // two Newton-Raphson steps y <- y + y (1 - x y^2) / 2, as above
  double y = rsqrt_approx(x);
  y = fma(0.5 * y, fma(-x * y, y, 1.0), y);
  return fma(0.5 * y, fma(-x * y, y, 1.0), y);
}

// Cholesky factor of a Hermitian matrix with dropped pivots, and the inverse of the factor, for
// n <= 32, by one warp without CTA barriers, in blocks of 8: the 8 x 8 diagonal block in registers (row lane % 8, values passed by
// shuffles), the panel rows below it one per lane, then the rank-8 update; after that lane c solves
// column c of L X = I block by block.  B (n x n, stride ld, lower triangle read and overwritten by
// L), X: the inverse (upper triangle zero), drop[j] set for pivots at or below tol, whose rows and
// columns become e_j.  The CTA-wide version spends such small sizes on barriers.
template <typename R>
__device__ void warp_chol_inverse(typename cplx_t<R>::type* B, typename cplx_t<R>::type* X, int n, int ld, R tol,
                                  int* drop) {
  typedef typename cplx_t<R>::type C2;
  constexpr int PB = 8;
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  for (int j0 = 0; j0 < n; j0 += PB) {
    const int jb = min(PB, n - j0), j1 = j0 + jb;
    const int r = lane & (PB - 1);
    C2 a[PB], b[PB];
    R inv[PB];
    const int i = j1 + lane;
#pragma unroll
    for (int c = 0; c < PB; ++c) {
      a[c] = (r < jb && c < jb) ? B[(j0 + r) * ld + j0 + c] : mk<R>(0, 0);
      b[c] = (i < n && c < jb) ? B[i * ld + j0 + c] : mk<R>(0, 0);
    }
#pragma unroll
    for (int j = 0; j < PB; ++j) {
      const R d = __shfl_sync(full, a[j].x, j);
      const bool keep = d > tol;
      if (j >= jb) { inv[j] = 0; continue; }
      const R is = inv_sqrt(d);
      inv[j] = keep ? is : (R)0;
      a[j] = r == j ? mk<R>(keep ? d * is : (R)1, 0) : cscale(a[j], inv[j]);
#pragma unroll
      for (int c = j + 1; c < PB; ++c) {
        const C2 lc = mk<R>(__shfl_sync(full, a[j].x, c), __shfl_sync(full, a[j].y, c));
        if (r >= c) {  // a_rc -= l_rj conj(l_cj)
          a[c].x -= a[j].x * lc.x + a[j].y * lc.y;
          a[c].y -= a[j].y * lc.x - a[j].x * lc.y;
        }
      }
    }
    if (j1 < n)
#pragma unroll
    for (int j = 0; j < PB; ++j) {
#pragma unroll
      for (int k = 0; k < j; ++k) {
        const C2 l = mk<R>(__shfl_sync(full, a[k].x, j), __shfl_sync(full, a[k].y, j));
        b[j].x -= b[k].x * l.x + b[k].y * l.y;
        b[j].y -= b[k].y * l.x - b[k].x * l.y;
      }
      b[j] = cscale(b[j], inv[j]);
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < PB; ++c) {
      if (c < jb && i < n) B[i * ld + j0 + c] = b[c];
      if (c < jb && lane < jb && c <= lane) B[(j0 + lane) * ld + j0 + c] = a[c];
      if (lane == c && c < jb) {
        X[(j0 + c) * ld + j0 + c].x = inv[c] == (R)0 ? (R)1 : inv[c];  // reciprocal diagonal, until X is formed
        if (inv[c] == (R)0) drop[j0 + c] = 1;
      }
    }
    __syncwarp();
    for (int c = j1; c < n; ++c) {
      if (i >= c && i < n) {
        C2 v = B[i * ld + c];
#pragma unroll
        for (int j = 0; j < PB; ++j) {  // rows remain below the panel only where it is full
          const C2 l = B[c * ld + j0 + j];
          v.x -= b[j].x * l.x + b[j].y * l.y;
          v.y -= b[j].y * l.x - b[j].x * l.y;
        }
        B[i * ld + c] = v;
      }
    }
    __syncwarp();
  }
  for (int i = 0; i < n; ++i)  // rows and columns of dropped coordinates
    if (lane < i && (drop[i] || drop[lane])) B[i * ld + lane] = mk<R>(0, 0);
  __syncwarp();
  // column `lane` of the inverse, top down
  for (int i0 = 0; i0 < n; i0 += PB) {
    const int ib = min(PB, n - i0);
    C2 x[PB];
#pragma unroll
    for (int q = 0; q < PB; ++q) x[q] = mk<R>(i0 + q == lane ? (R)1 : (R)0, 0);
    R id[PB];
#pragma unroll
    for (int q = 0; q < PB; ++q) id[q] = X[min(i0 + q, n - 1) * (ld + 1)].x;
    __syncwarp();
    if (lane < n) {
      for (int k = 0; k < i0; ++k) {
        const C2 xk = X[k * ld + lane];
#pragma unroll
        for (int q = 0; q < PB; ++q) {
          const C2 l = B[min(i0 + q, n - 1) * ld + k];
          cfma(x[q], mk<R>(-l.x, -l.y), xk);
        }
      }
#pragma unroll
      for (int q = 0; q < PB; ++q) {
        if (q < ib) {
#pragma unroll
          for (int k = 0; k < q; ++k) {
            const C2 l = B[(i0 + q) * ld + i0 + k];
            cfma(x[q], mk<R>(-l.x, -l.y), x[k]);
          }
          x[q] = cscale(x[q], id[q]);
          X[(i0 + q) * ld + lane] = lane <= i0 + q ? x[q] : mk<R>(0, 0);
        }
      }
    }
  }
  __syncwarp();
}

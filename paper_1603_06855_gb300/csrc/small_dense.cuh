// Small dense Hermitian algebra in shared memory for one CTA (any block size): Cholesky with
// column dropping and the in-place inverse of a lower-triangular factor.  Shared by the
// projected-problem kernels of both precisions.
#pragma once
#include "kernels.h"

// Cholesky of Hermitian B (n x n, stride ld) with column dropping, in place (lower
// triangle); drop[j] = 1 for a pivot at or below tol (dropped rows/columns become e_j).
template <typename R>
__device__ void chol_drop(typename cplx_t<R>::type* B, int n, int ld, R tol, int* drop) {
  typedef typename cplx_t<R>::type C2;
  for (int j = 0; j < n; ++j) {
    __syncthreads();
    R d = B[j * ld + j].x;
    bool dr = !(d > tol);
    __syncthreads();
    if (dr) {
      for (int i = threadIdx.x; i < n; i += blockDim.x)
        if (i != j) { B[i * ld + j] = mk<R>(0, 0); B[j * ld + i] = mk<R>(0, 0); }
      if (threadIdx.x == 0) { B[j * ld + j] = mk<R>(1, 0); drop[j] = 1; }
      continue;
    }
    R sq = sqrt(d), inv = (R)1 / sq;
    for (int i = j + 1 + threadIdx.x; i < n; i += blockDim.x) B[i * ld + j] = cscale(B[i * ld + j], inv);
    if (threadIdx.x == 0) B[j * ld + j] = mk<R>(sq, 0);
    __syncthreads();
    int nt = n - j - 1;
    for (int t = threadIdx.x; t < nt * nt; t += blockDim.x) {
      int i = j + 1 + t / nt, c = j + 1 + t % nt;
      if (c <= i) {
        C2 v = B[i * ld + c];
        C2 l1 = B[i * ld + j], l2 = B[c * ld + j];
        v.x -= l1.x * l2.x + l1.y * l2.y;
        v.y -= l1.y * l2.x - l1.x * l2.y;
        B[i * ld + c] = v;
      }
    }
  }
  __syncthreads();
}

// In-place inverse of the lower-triangular L (n x n, stride ld); upper triangle zeroed.
// Column j of the inverse from columns j+1.. (already inverted): one warp per row, lanes
// split the dot product and reduce with shuffles.
template <typename R>
__device__ void tri_inv_lower(typename cplx_t<R>::type* L, int n, int ld, typename cplx_t<R>::type* tmp) {
  typedef typename cplx_t<R>::type C2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int j = n - 1; j >= 0; --j) {
    __syncthreads();
    C2 ljj = L[j * ld + j];
    R den = ljj.x * ljj.x + ljj.y * ljj.y;
    C2 ajj = mk<R>(ljj.x / den, -ljj.y / den);
    for (int i = j + 1 + threadIdx.x; i < n; i += blockDim.x) tmp[i] = L[i * ld + j];
    __syncthreads();
    // new L[i][j] = -ajj * sum_{c=j+1..i} Linv[i][c] * old L[c][j]
    for (int i = j + 1 + warp; i < n; i += nw) {
      C2 s = mk<R>(0, 0);
      for (int c = j + 1 + lane; c <= i; c += 32) cfma(s, L[i * ld + c], tmp[c]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
      }
      if (lane == 0) {
        C2 v = cmul(s, ajj);
        L[i * ld + j] = mk<R>(-v.x, -v.y);
      }
    }
    if (threadIdx.x == 0) L[j * ld + j] = ajj;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    int i = t / n, c = t % n;
    if (c > i) L[i * ld + c] = mk<R>(0, 0);
  }
  __syncthreads();
}

// The same factorisation and the inverse of its factor for n <= 32, by one warp without CTA
// barriers, in blocks of 8: the 8 x 8 diagonal block in registers (row lane % 8, values passed by
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
      const R sq = sqrt(d);
      inv[j] = keep ? (R)1 / sq : (R)0;
      a[j] = r == j ? mk<R>(keep ? sq : (R)1, 0) : cscale(a[j], inv[j]);
#pragma unroll
      for (int c = j + 1; c < PB; ++c) {
        const C2 lc = mk<R>(__shfl_sync(full, a[j].x, c), __shfl_sync(full, a[j].y, c));
        if (r >= c) {  // a_rc -= l_rj conj(l_cj)
          a[c].x -= a[j].x * lc.x + a[j].y * lc.y;
          a[c].y -= a[j].y * lc.x - a[j].x * lc.y;
        }
      }
    }
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
      if (lane == c && c < jb && inv[c] == (R)0) drop[j0 + c] = 1;
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
          x[q] = cscale(x[q], (R)1 / B[(i0 + q) * ld + i0 + q].x);
          X[(i0 + q) * ld + lane] = lane <= i0 + q ? x[q] : mk<R>(0, 0);
        }
      }
    }
  }
  __syncwarp();
}

// Small dense Hermitian eigenproblems in shared memory, one CTA per problem (n <= 72), for both
// precisions: the pieces of the projected-problem kernels (small_rr.cu, small_rr64.cu).
#pragma once
#include "kernels.h"
#include "small_dense.cuh"

constexpr int SR_NMAX = 72;
constexpr int SR_LD = 74;                       // even row stride: 16-byte aligned element pairs
constexpr int SR_MAT = SR_NMAX * SR_LD;         // complex elements per matrix
constexpr int SR_MAX_SWEEPS = 16;               // 5 to 7 are taken

// Complex arithmetic with explicit roundings, so that every call site computes bitwise the
// same value from the same inputs (the plane threads recompute entries the block threads
// store).
__device__ __forceinline__ float2 zmul(float2 a, float2 b) {
  return make_float2(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x)));
}
__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(__fma_rn(a.x, b.x, -__dmul_rn(a.y, b.y)), __fma_rn(a.x, b.y, __dmul_rn(a.y, b.x)));
}
// c x + z (c real)
__device__ __forceinline__ float2 zaxpy(float c, float2 x, float2 z) {
  return make_float2(__fmaf_rn(c, x.x, z.x), __fmaf_rn(c, x.y, z.y));
}
__device__ __forceinline__ double2 zaxpy(double c, double2 x, double2 z) {
  return make_double2(__fma_rn(c, x.x, z.x), __fma_rn(c, x.y, z.y));
}
template <typename C2> __device__ __forceinline__ C2 zneg(C2 a) { a.x = -a.x; a.y = -a.y; return a; }
// conj(a) where f
template <typename C2> __device__ __forceinline__ C2 conj_if(C2 a, bool f) { if (f) a.y = -a.y; return a; }

// Rotation of a plane: col_u <- c col_u - conj(s) col_v, col_v <- s col_u + c col_v; on: s != 0.
template <typename R> struct __align__(16) Plane {
  typename cplx_t<R>::type s;
  R c;
  int on;
};

// Entry (r, col) of J1^H M J2 for a 2 x 2 block M (rows: plane 1, columns: plane 2) from the entries
// named relative to it: ms[a] = M[a == 0 ? r : 1 - r][col], mo[a] the same rows' other column.
// sg2 = -1 for col = 0, +1 for col = 1; sg1 the same of r.
template <typename R, typename C2 = typename cplx_t<R>::type>
__device__ __forceinline__ C2 rotated(C2 ms0, C2 mo0, C2 ms1, C2 mo1, const Plane<R>& p1, R sg1, const Plane<R>& p2, R sg2) {
  const C2 s2 = mk<R>(sg2 * p2.s.x, p2.s.y);    // -conj(s) or s
  const C2 y0 = zaxpy(p2.c, ms0, zmul(s2, mo0)), y1 = zaxpy(p2.c, ms1, zmul(s2, mo1));
  const C2 s1 = mk<R>(sg1 * p1.s.x, -p1.s.y);   // -s or conj(s)
  return zaxpy(p1.c, y0, zmul(s1, y1));
}

// Next position of the circle method in pair-ordered positions (top[t] = 2t, bottom[t] = 2t+1):
// top[0] stays, top[t] -> top[t+1], top[np-1] -> bottom[np-1], bottom[t] -> bottom[t-1],
// bottom[0] -> top[1].  One cycle through the 2 np - 1 moving positions.
__device__ __forceinline__ int next_pos(int pos, int np) {
  if (np == 1 || pos == 0) return pos;
  if (pos & 1) return pos == 1 ? 2 : pos - 2;
  return (pos >> 1) == np - 1 ? pos + 1 : pos + 2;
}
__device__ __forceinline__ int prev_pos(int pos, int np) {
  if (np == 1 || pos == 0) return pos;
  if (pos & 1) return pos == 2 * np - 1 ? pos - 1 : pos + 2;
  return pos == 2 ? 1 : pos - 2;
}

// Element (i, j) of the rotated matrix in its buffer: the even (top) columns of a row, then the odd
// ones, so that neighbouring planes' entries are neighbours both where they are read and, shifted
// by one plane, where they are written: no bank conflicts on either side.
__device__ __forceinline__ int spos(int i, int j) { return i * SR_LD + (j & 1) * (SR_LD / 2) + (j >> 1); }

__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Whether the plane of entries a_uu, a_vv (real) and a_uv rotates.  (A plane of the padding
// coordinate, whose row and column are zero and stay zero, never does.)
__device__ __forceinline__ bool plane_rotates(float app, float aqq, float b2, float floor_abs) {
  return sqrt_approx(b2) > 1.1920929e-07f * sqrt_approx(fabsf(app * aqq)) + floor_abs;
}

// Rotation of the plane of positions (u, v) from a_uu, a_vv (real) and a_uv:
// with d = a_vv - a_uu and b = |a_uv|, t = 2 b sgn(d) / (|d| + sqrt(d^2 + 4 b^2)) is the tangent
// of the smaller rotation angle, c = 1 / sqrt(1 + t^2) and s = c t a_uv / b.  The chain of a round
// runs through here, so it has no branch, and the root and reciprocal are the hardware
// approximations: their error (a few units in the last place) turns the angle by as little, which
// only leaves that share of a_uv, below its rounding.  c comes from the tangent that is used, as
// 1 - t^2 r(t^2) with r(x) = 1 / (1 + x + sqrt(1 + x)) on [0, 1] (its Chebyshev interpolant of degree 9,
// 5e-8 relative): an error of r counts by t^2 only, so c^2 + |s|^2 = 1 holds to rounding also for the
// many small rotations of the last sweeps (with the approximate reciprocal root and a Newton step
// the columns' norms drifted by 1e-5 over a solve).
__device__ __forceinline__ Plane<float> make_plane(float app, float aqq, float2 apq, float floor_abs) {
  const float b2 = __fmaf_rn(apq.x, apq.x, apq.y * apq.y);
  const bool on = plane_rotates(app, aqq, b2, floor_abs);
  const float d = aqq - app;
  const float inv = rcp_approx(fabsf(d) + sqrt_approx(__fmaf_rn(d, d, 4.f * b2)));
  const float g = 2.f * inv;                     // |tangent| / b
  const float x = g * g * b2, x2 = x * x, x4 = x2 * x2;
  const float r01 = __fmaf_rn(-0.37499827f, x, 0.5f), r23 = __fmaf_rn(-0.2726586f, x, 0.31244183f);
  const float r45 = __fmaf_rn(-0.20286512f, x, 0.24065118f), r67 = __fmaf_rn(-0.08192697f, x, 0.14801665f);
  const float r89 = __fmaf_rn(-0.00477741f, x, 0.02900993f);
  const float r0 = __fmaf_rn(r23, x2, r01), r4 = __fmaf_rn(r67, x2, r45);
  const float c = 1.f - x * __fmaf_rn(__fmaf_rn(r89, x4, r4), x4, r0);
  const float f = (d >= 0.f ? g : -g) * c;       // c t / b
  Plane<float> w;
  w.c = on ? c : 1.f;
  w.s = make_float2(on ? f * apq.x : 0.f, on ? f * apq.y : 0.f);
  w.on = on ? 1 : 0;
  return w;
}

// The same in FP64.  The hardware's FP64 root and reciprocal approximations carry some 20 bits; one
// Newton-Raphson step each gives the angle to about 1e-12, and what that leaves of a_uv goes to the next
// sweep (the entry is not set to zero).  c = (1 + t^2)^-1/2 is exact to rounding for the tangent used: its
// binomial series for small t^2 (all but a few rotations here), else the correctly rounded root.
__device__ __forceinline__ bool plane_rotates(double app, double aqq, double b2, double floor_abs) {
  const double x = fabs(app * aqq);
  const double t = x > 0.0 ? fma(2.220446049250313e-16 * x, rsqrt_approx(x), floor_abs) : floor_abs;
  return b2 > t * t;
}
__device__ __forceinline__ Plane<double> make_plane(double app, double aqq, double2 apq, double floor_abs) {
  const double b2 = fma(apq.x, apq.x, apq.y * apq.y);
  Plane<double> w;
  w.c = 1.0;
  w.s = make_double2(0.0, 0.0);
  w.on = 0;
  if (plane_rotates(app, aqq, b2, floor_abs)) {
    const double d = aqq - app;
    const double v = fma(d, d, 4.0 * b2);
    double y = rsqrt_approx(v);
    y = fma(0.5 * y, fma(-v * y, y, 1.0), y);
    const double den = fma(v, y, fabs(d));
    double inv = rcp_approx(den);
    inv = fma(inv, fma(-den, inv, 1.0), inv);
    const double g = 2.0 * inv;                  // |tangent| / b
    const double x = g * g * b2;
    double c;
    if (x < 1e-3) {
      c = fma(x, 231.0 / 1024.0, -63.0 / 256.0);
      c = fma(c, x, 35.0 / 128.0);
      c = fma(c, x, -5.0 / 16.0);
      c = fma(c, x, 3.0 / 8.0);
      c = fma(c, x, -0.5);
      c = fma(c, x, 1.0);
    } else {
      c = 1.0 / sqrt(1.0 + x);
    }
    const double f = (d >= 0.0 ? g : -g) * c;    // c t / b
    w.c = c;
    w.s = make_double2(f * apq.x, f * apq.y);
    w.on = 1;
  }
  return w;
}

// Barrier over the first `threads` threads of the CTA (a multiple of 32), and the same with an OR.
__device__ __forceinline__ void bar_first(int threads) {
  asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
}
__device__ __forceinline__ bool bar_first_or(int threads, bool p) {
  int r;
  asm volatile(
      "{\n\t.reg .pred q, w;\n\tsetp.ne.s32 q, %2, 0;\n\tbar.red.or.pred w, 1, %1, q;\n\tselp.s32 %0, 1, 0, w;\n\t}"
      : "=r"(r)
      : "r"(threads), "r"((int)p)
      : "memory");
  return r != 0;
}

// Cholesky of the Hermitian B (lower, row stride SR_LD) with dropped pivots; invd: the reciprocal
// diagonal.  On return dropped rows and columns are e_j.
template <typename R, int PB, int THREADS, typename C2 = typename cplx_t<R>::type>
__device__ __forceinline__ void block_cholesky(C2* B, int n, R drop_tol, int* drop, R* invd) {
  constexpr int W = THREADS / 32;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int j0 = 0; j0 < n; j0 += PB) {
    const int jb = min(PB, n - j0), j1 = j0 + jb;
    C2 a[PB];
    if (warp == 0 || j1 + 32 * warp < n) {
      // every warp with panel rows factors the diagonal block (row lane % PB) for itself
      const int r = lane & (PB - 1);
      R inv[PB];
#pragma unroll
      for (int c = 0; c < PB; ++c) a[c] = (r < jb && c < jb) ? B[(j0 + r) * SR_LD + j0 + c] : mk<R>(0, 0);
#pragma unroll
      for (int j = 0; j < PB; ++j) {
        const R d = __shfl_sync(0xffffffffu, a[j].x, j);
        const bool keep = d > drop_tol;
        const R is = inv_sqrt(d);
        inv[j] = keep ? is : (R)0;
        if (r == j) a[j] = mk<R>(keep ? d * is : (R)1, (R)0);
        else a[j] = mk<R>(a[j].x * inv[j], a[j].y * inv[j]);
#pragma unroll
        for (int c = j + 1; c < PB; ++c) {
          const C2 lc = mk<R>(__shfl_sync(0xffffffffu, a[j].x, c), __shfl_sync(0xffffffffu, a[j].y, c));
          if (r >= c) {  // a_rc -= l_rj conj(l_cj)
            a[c].x -= a[j].x * lc.x + a[j].y * lc.y;
            a[c].y -= a[j].y * lc.x - a[j].x * lc.y;
          }
        }
      }
      const int i = j1 + 32 * warp + lane;
      C2 b[PB];
#pragma unroll
      for (int c = 0; c < PB; ++c) b[c] = i < n && c < jb ? B[i * SR_LD + j0 + c] : mk<R>(0, 0);
#pragma unroll
      for (int j = 0; j < PB; ++j) {
#pragma unroll
        for (int k = 0; k < j; ++k) {
          const C2 l = mk<R>(__shfl_sync(0xffffffffu, a[k].x, j), __shfl_sync(0xffffffffu, a[k].y, j));
          b[j].x -= b[k].x * l.x + b[k].y * l.y;
          b[j].y -= b[k].y * l.x - b[k].x * l.y;
        }
        b[j].x *= inv[j];
        b[j].y *= inv[j];
      }
      if (i < n)
#pragma unroll
        for (int c = 0; c < PB; ++c)
          if (c < jb) B[i * SR_LD + j0 + c] = b[c];
      if (warp == 0)
#pragma unroll
        for (int c = 0; c < PB; ++c)
          if (lane == c && c < jb) {
            drop[j0 + c] = inv[c] == (R)0 ? 1 : 0;
            invd[j0 + c] = inv[c] == (R)0 ? (R)1 : inv[c];
          }
    }
    __syncthreads();
    if (warp == 0 && lane < jb)  // every warp has read the diagonal block
#pragma unroll
      for (int c = 0; c < PB; ++c)
        if (c <= lane) B[(j0 + lane) * SR_LD + j0 + c] = a[c];
    // trailing update of the rows and columns from j1 on by the panel (dropped columns are zero)
    const int nt = n - j1;
    for (int rr = warp; rr < nt; rr += W) {
      const int i = j1 + rr;
      for (int q = lane; q <= rr; q += 32) {
        const int c = j1 + q;
        C2 v = B[i * SR_LD + c];
#pragma unroll
        for (int h = 0; h < PB; h += 2) {  // the panel is full wherever rows remain below it
          C2 x0, x1, y0, y1;
          if constexpr (sizeof(R) == 4) {  // two entries per load
            const float4 x = *reinterpret_cast<const float4*>(B + i * SR_LD + j0 + h);
            const float4 y = *reinterpret_cast<const float4*>(B + c * SR_LD + j0 + h);
            x0 = mk<R>(x.x, x.y); x1 = mk<R>(x.z, x.w); y0 = mk<R>(y.x, y.y); y1 = mk<R>(y.z, y.w);
          } else {
            x0 = B[i * SR_LD + j0 + h]; x1 = B[i * SR_LD + j0 + h + 1];
            y0 = B[c * SR_LD + j0 + h]; y1 = B[c * SR_LD + j0 + h + 1];
          }
          v.x -= x0.x * y0.x + x0.y * y0.y;
          v.y -= x0.y * y0.x - x0.x * y0.y;
          v.x -= x1.x * y1.x + x1.y * y1.y;
          v.y -= x1.y * y1.x - x1.x * y1.y;
        }
        B[i * SR_LD + c] = v;
      }
    }
    __syncthreads();
  }
  for (int i = warp; i < n; i += W)
    for (int c = lane; c <= i; c += 32)
      if (drop[i] || drop[c]) B[i * SR_LD + c] = mk<R>(i == c ? (R)1 : (R)0, (R)0);
  __syncthreads();
}

// Forward substitution L X = R in place, right-looking in blocks of PB rows.  Columns c < n0 of R are
// columns of P0, the others columns c - n0 of P1.  tri = 1: P1 starts as the identity, whose
// column j is zero above row j; tri = 2 (n0 = ncol): only rows i <= c of column c are wanted.
template <typename R, int PB, int THREADS, typename C2 = typename cplx_t<R>::type>
__device__ __forceinline__ void block_forward(const C2* L, const R* invd, C2* P0, C2* P1, int n0, int n, int ncol, int tri) {
  const int tid = threadIdx.x;
  for (int i0 = 0; i0 < n; i0 += PB) {
    const int ib = min(PB, n - i0), i1 = i0 + ib;
    const int c_lo = tri == 2 ? i0 : 0;
    const int c_hi = tri == 1 ? n0 + min(n, i1) : ncol;
    for (int c = c_lo + tid; c < c_hi; c += THREADS) {
      C2* X = c < n0 ? P0 + c : P1 + (c - n0);
      C2 x[PB];
#pragma unroll
      for (int ii = 0; ii < PB; ++ii) {
        if (ii < ib) {
          const int i = i0 + ii;
          C2 acc = X[i * SR_LD];
#pragma unroll
          for (int kk = 0; kk < ii; ++kk) {
            const C2 l = L[i * SR_LD + i0 + kk];
            acc.x -= l.x * x[kk].x - l.y * x[kk].y;
            acc.y -= l.x * x[kk].y + l.y * x[kk].x;
          }
          x[ii] = mk<R>(acc.x * invd[i], acc.y * invd[i]);
          X[i * SR_LD] = x[ii];
        }
      }
    }
    __syncthreads();
    if (i1 >= n) break;
    // rows below: four rows of one column per thread (i1 is a multiple of 4 here)
    const int nc = c_hi - c_lo, ng = (n - i1 + 3) / 4;
    for (int e = tid; e < nc * ng; e += THREADS) {
      const int g = e / nc, c = c_lo + e - g * nc;
      const int r0 = i1 + 4 * g;
      if (tri == 2 && c < r0) continue;
      C2* X = c < n0 ? P0 + c : P1 + (c - n0);
      C2 acc[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] = mk<R>(0, 0);
#pragma unroll
      for (int k = 0; k < PB; ++k) {
        const C2 x = X[(i0 + k) * SR_LD];
#pragma unroll
        for (int q = 0; q < 4; ++q) cfma(acc[q], L[(r0 + q) * SR_LD + i0 + k], x);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (r0 + q < n) X[(r0 + q) * SR_LD] = csub(X[(r0 + q) * SR_LD], acc[q]);
    }
    __syncthreads();
  }
}

// Backward substitution L^H X = W in place for ncol columns (row stride ldw).
template <typename R, int PB, int THREADS, typename C2 = typename cplx_t<R>::type>
__device__ __forceinline__ void block_backward(const C2* L, C2* W, int ldw, int n, int ncol) {
  const int tid = threadIdx.x;
  for (int i0 = ((n - 1) / PB) * PB; i0 >= 0; i0 -= PB) {
    const int ib = min(PB, n - i0);
    for (int c = tid; c < ncol; c += THREADS) {
      C2 x[PB];
#pragma unroll
      for (int ii = PB - 1; ii >= 0; --ii) {
        if (ii < ib) {
          C2 acc = W[(i0 + ii) * ldw + c];
#pragma unroll
          for (int kk = ii + 1; kk < PB; ++kk)
            if (kk < ib) acc = csub(acc, cmulc(L[(i0 + kk) * SR_LD + i0 + ii], x[kk]));
          x[ii] = cscale(acc, (R)1 / L[(i0 + ii) * SR_LD + i0 + ii].x);
          W[(i0 + ii) * ldw + c] = x[ii];
        }
      }
    }
    __syncthreads();
    for (int e = tid; e < i0 * ncol; e += THREADS) {
      const int r = e / ncol, c = e - r * ncol;
      C2 acc = W[r * ldw + c];
      for (int k = 0; k < ib; ++k) acc = csub(acc, cmulc(L[(i0 + k) * SR_LD + r], W[(i0 + k) * ldw + c]));
      W[r * ldw + c] = acc;
    }
    __syncthreads();
  }
}

// Cyclic two-sided Jacobi on the position-ordered matrix in Sa (layout spos, upper triangle; Sb: the
// second buffer), nk_ coordinates padded to 2 np.  Roles by warp, in this order: pw plane warps (ten
// planes of three lanes each) and bw block warps (one 2 x 2 block of the upper triangle per thread).
// Only these take part in the rounds' barriers; the rest wait at the end.  S is in Sa in even rounds
// and Sb in odd ones.  pl: 2 x 36 planes; the planes of every round are logged to logk, np a round.
// Only the m lowest eigenpairs are wanted: after a sweep (every index is back at its own position) the
// iteration has converged when no pair with one of the m smallest diagonal entries would rotate and
// the other pairs are below 1e-3 of sqrt(a_ii a_jj), which keeps the eigenvalues among them away from
// the lowest (each within 7 % of a diagonal entry for n <= 72).  With `correct` a wanted pair may also
// be left to the first-order correction v_j = e_j + sum_i a_ij / (a_jj - a_ii) e_i, which replay() starts
// from, where its term is at most JacTol::first sqrt(ratio of the two entries) and the other pairs are
// below JacTol::rest: what the correction leaves out, the term times the coupling of the rest, then
// stays below the rounding in every coordinate relative to its own size.  (Without the ratio, 1e-7 of a
// direction whose Rayleigh quotient is 800 times larger came through, and single k-points of
// high-contrast cells settled at residuals of 3e-3.)  The two save one of six sweeps against asking the
// test of all pairs.  On return ev holds the diagonal and perm the positions by ascending entry; the
// last matrix is in Sa after an even number of rounds, else in Sb.  Returns the number of sweeps.
template <typename R> struct JacTol;
template <> struct JacTol<float> { static constexpr float rest = 1e-4f, first = 5e-5f; };
template <> struct JacTol<double> { static constexpr double rest = 1e-8, first = 1e-9; };
// The correction term a_ij / (a_jj - a_ii), and whether it is small enough to replace the rotation.
template <typename R, typename C2 = typename cplx_t<R>::type>
__device__ __forceinline__ bool pair_corrects(R aii, R ajj, C2 aij, C2& v) {
  const R x = fabs(aii), y = fabs(ajj), gap = ajj - aii;
  if (gap == (R)0) return false;
  v = mk<R>(aij.x / gap, aij.y / gap);
  return (v.x * v.x + v.y * v.y) * fmax(x, y) <= JacTol<R>::first * JacTol<R>::first * fmin(x, y);
}
template <typename R, int THREADS, typename C2 = typename cplx_t<R>::type>
__device__ __forceinline__ int jacobi_sweeps(C2* Sa, C2* Sb, Plane<R>* pl, Plane<R>* __restrict__ logk, int nk_, int m,
                                             R floor_abs, bool correct, R* ev, int* perm, int* low, int* misc) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int npad = nk_ + (nk_ & 1), np = npad / 2, nrounds = npad - 1;
  const int nblk = np * (np + 1) / 2;
  if (tid < np) {  // planes of the first round
    const int u = 2 * tid, v = u + 1;
    const Plane<R> w = make_plane(Sa[spos(u, u)].x, Sa[spos(v, v)].x, Sa[spos(u, v)], floor_abs);
    pl[tid] = w;
    logk[tid] = w;
  }
  __syncthreads();
  const int pw = (np + 9) / 10, bw = (nblk + 31) / 32;
  const int nact = 32 * (pw + bw);
  int sweeps = 0, par = 0;
  auto more = [&]() {
    ++sweeps;
    const C2* S = par ? Sb : Sa;
    for (int p = tid; p < nk_; p += nact) {
      ev[p] = S[spos(p, p)].x;
      perm[p] = p;  // stays where a NaN leaves ranks open
    }
    bar_first(nact);
    for (int p = tid; p < nk_; p += nact) {
      int r = 0;
      const R vi = ev[p];
      for (int q = 0; q < nk_; ++q) r += (ev[q] < vi || (ev[q] == vi && q < p)) ? 1 : 0;
      perm[r] = p;
      low[p] = r < m ? 1 : 0;
    }
    bar_first(nact);
    bool any = false, left = false, rest = false;
    for (int i = warp; i < nk_; i += nact / 32) {
      const R aii = ev[i];
      const int li = low[i];
      for (int j = i + 1 + lane; j < nk_; j += 32) {
        const C2 a = S[spos(i, j)];
        const R b2 = a.x * a.x + a.y * a.y;
        if (li | low[j]) {
          if (plane_rotates(aii, ev[j], b2, floor_abs)) {
            C2 v;
            if (correct && pair_corrects<R>(aii, ev[j], a, v)) left = true;
            else any = true;
          }
        } else {
          const R d2 = fabs(aii * ev[j]);
          any |= b2 > (R)1e-6 * d2 + floor_abs * floor_abs;
          rest |= b2 > JacTol<R>::rest * JacTol<R>::rest * d2 + floor_abs * floor_abs;
        }
      }
    }
    if (sweeps >= SR_MAX_SWEEPS) return false;
    if (bar_first_or(nact, any)) return true;
    return bar_first_or(nact, left) && bar_first_or(nact, rest);
  };
  if (warp < pw) {
    // plane pt of the next round from the entries at its positions u0, v0 of this one:
    // pe = 0: a_uu, 1: a_vv, 2: a_uv
    const int pt = warp * 10 + lane / 3, pe = lane % 3, pbase = lane - pe;
    const bool mine = lane < 30 && pt < np;
    int l0 = 0, l1 = 0, l2 = 0, l3 = 0, t1 = 0, t2 = 0;
    bool g0 = false, g1 = false, g2 = false, g3 = false, ge = false;
    R sg1 = 0, sg2 = 0;
    if (mine) {
      const int u0 = prev_pos(2 * pt, np), v0 = prev_pos(2 * pt + 1, np);
      int u = pe == 1 ? v0 : u0, v = pe == 0 ? u0 : v0;
      if ((u >> 1) > (v >> 1)) {  // the stored block is the transposed one: conjugate the result
        const int x = u;
        u = v;
        v = x;
        ge = true;
      }
      t1 = u >> 1;
      t2 = v >> 1;
      const int r = u & 1, c = v & 1;
      sg1 = r ? (R)1 : (R)-1;
      sg2 = c ? (R)1 : (R)-1;
      // entries M[r][c], M[r][1-c], M[1-r][c], M[1-r][1-c]; below the diagonal the conjugate above it
      auto at = [&](int rr, int cc, bool& f) {
        const int i = 2 * t1 + rr, j = 2 * t2 + cc;
        f = i > j;
        return i <= j ? spos(i, j) : spos(j, i);
      };
      l0 = at(r, c, g0);
      l1 = at(r, 1 - c, g1);
      l2 = at(1 - r, c, g2);
      l3 = at(1 - r, 1 - c, g3);
    }
    Plane<R>* log_next = logk + np;
    do {
      for (int round = 0; round < nrounds; ++round) {
        const C2* S = par ? Sb : Sa;
        const Plane<R>* cur = pl + par * 36;
        const Plane<R> p1 = cur[t1], p2 = cur[t2];
        C2 e = rotated<R>(conj_if(S[l0], g0), conj_if(S[l1], g1), conj_if(S[l2], g2), conj_if(S[l3], g3), p1, sg1, p2, sg2);
        if constexpr (sizeof(R) == 4) {
          if (np == 1 && p1.on) e = mk<R>(pe == 2 ? (R)0 : e.x, (R)0);  // its own plane annihilated it
        }
        e = conj_if(e, ge);
        const R auu = __shfl_sync(0xffffffffu, e.x, pbase & 31);
        const R avv = __shfl_sync(0xffffffffu, e.x, (pbase + 1) & 31);
        const C2 auv = mk<R>(__shfl_sync(0xffffffffu, e.x, (pbase + 2) & 31),
                             __shfl_sync(0xffffffffu, e.y, (pbase + 2) & 31));
        if (mine && pe == 0) {
          const Plane<R> w = make_plane(auu, avv, auv, floor_abs);
          pl[(par ^ 1) * 36 + pt] = w;
          log_next[pt] = w;
        }
        log_next += np;
        bar_first(nact);
        par ^= 1;
      }
    } while (more());
    if (tid == 0) misc[3] = sweeps;
  } else if (warp < pw + bw) {
    const int u = tid - 32 * pw;
    const bool mine = u < nblk;
    int t1 = 0, t2 = 0, l0 = 0, w0 = 0, w1 = 0, w2 = 0, w3 = 0;
    bool f0 = false, f1 = false, f2 = false, f3 = false;
    if (mine) {
      int rem = u;
      while (rem >= np - t1) { rem -= np - t1; ++t1; }
      t2 = t1 + rem;
      l0 = spos(2 * t1, 2 * t2);
      const int ra = next_pos(2 * t1, np), rb = next_pos(2 * t1 + 1, np);
      const int ca = next_pos(2 * t2, np), cb = next_pos(2 * t2 + 1, np);
      auto to = [&](int i, int j, bool& f) {
        f = i > j;
        return i <= j ? spos(i, j) : spos(j, i);
      };
      w0 = to(ra, ca, f0);
      w1 = to(ra, cb, f1);
      w2 = to(rb, ca, f2);
      w3 = to(rb, cb, f3);
    }
    const bool dg = t1 == t2;
    do {
      for (int round = 0; round < nrounds; ++round) {
        if (mine) {
          const C2* S = par ? Sb : Sa;
          C2* T = par ? Sa : Sb;
          const Plane<R>* cur = pl + par * 36;
          const Plane<R> p1 = cur[t1], p2 = cur[t2];
          const C2 m00 = S[l0], m01 = S[l0 + SR_LD / 2], m11 = S[l0 + SR_LD + SR_LD / 2];
          C2 m10 = S[l0 + SR_LD];
          if (dg) m10 = cconj(m01);
          C2 e00 = rotated<R>(m00, m01, m10, m11, p1, (R)-1, p2, (R)-1);
          C2 e01 = rotated<R>(m01, m00, m11, m10, p1, (R)-1, p2, (R)1);
          const C2 e10 = rotated<R>(m10, m11, m00, m01, p1, (R)1, p2, (R)-1);
          C2 e11 = rotated<R>(m11, m10, m01, m00, p1, (R)1, p2, (R)1);
          if (dg) {
            e00.y = 0;
            e11.y = 0;
            if constexpr (sizeof(R) == 4) {
              if (p1.on) e01 = mk<R>(0, 0);
            }
          } else {
            T[w2] = conj_if(e10, f2);
          }
          T[w0] = conj_if(e00, f0);
          T[w1] = conj_if(e01, f1);
          T[w3] = conj_if(e11, f3);
        }
        bar_first(nact);
        par ^= 1;
      }
    } while (more());
  }
  __syncthreads();
  return misc[3];
}

// Eigenvectors of the packed matrix from the logged rotations (np planes per round, K rounds):
// column j < ncols of Y (nk_ rows, stride ldy) = J_1 P_1 J_2 P_2 ... J_K P_K e, e the unit vector of
// position perm[j] (with the first-order correction of jacobi_sweeps from the last matrix Sf and its
// diagonal ev, where given), P the circle method's moves.  Applied to the wanted columns only, from the last
// round back, which for n / 3 columns is a third of the work of accumulating all of V beside the
// rotations and leaves the shared-memory bandwidth of the rounds to the matrix (it was their bound
// in FP32: 147 KB a round at n = 69, of which V took 87).  LANES lanes hold a column, PPL planes
// (2 PPL positions) each, in registers; a move is one complex value from each neighbouring lane.  The
// last warps bring the log from L2 in chunks of SR_CHUNK rounds, one ahead.
constexpr int SR_CHUNK = 64;  // rounds x 36 planes x 16 (FP32) or 32 bytes: 36 or 72 KB per buffer
template <typename R, int LANES, int PPL, int THREADS, typename C2 = typename cplx_t<R>::type>
__device__ __forceinline__ void replay(const Plane<R>* __restrict__ logk, int K, int np, int nk_, int ncols,
                                       const int* perm, Plane<R>* buf0, Plane<R>* buf1, C2* Y, int ldy,
                                       const C2* Sf = nullptr, const R* ev = nullptr) {
  constexpr int PER = 32 / LANES, V = sizeof(Plane<R>) / 16;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int hl = lane % LANES;
  const int nchunk = (K + SR_CHUNK - 1) / SR_CHUNK;
  auto bring = [&](int c, int first, int step) {  // rounds c SR_CHUNK .. of the log
    float4* dst = reinterpret_cast<float4*>((c & 1) ? buf1 : buf0);
    const int cnt = min(SR_CHUNK, K - c * SR_CHUNK) * np * V;
    const float4* src = reinterpret_cast<const float4*>(logk + (long long)c * SR_CHUNK * np);
#pragma unroll 4
    for (int e = first; e < cnt; e += step) dst[e] = __ldcg(src + e);
  };
  int tp[PPL];       // plane read (those past the last hold nothing: their values reach no column)
  bool last[PPL];
  const bool first = hl == 0;
#pragma unroll
  for (int b = 0; b < PPL; ++b) {
    tp[b] = min(hl * PPL + b, np - 1);
    last[b] = hl * PPL + b == np - 1;
  }
  for (int c0 = 0; c0 < ncols;) {
    const int cw = min((ncols - c0 + PER - 1) / PER, THREADS / 32 - 1);  // warps that hold columns
    const int j = c0 + PER * warp + lane / LANES;
    const bool col = warp < cw;
    C2 top[PPL], bot[PPL];
    const int pj = col && j < ncols ? perm[j] : -1;
#pragma unroll
    for (int b = 0; b < PPL; ++b) {
      const int t = hl * PPL + b;
      auto start = [&](int p) {
        if (p == pj) return mk<R>((R)1, (R)0);
        if (!Sf || pj < 0 || p >= nk_) return mk<R>((R)0, (R)0);
        const C2 a = p < pj ? Sf[spos(p, pj)] : cconj(Sf[spos(pj, p)]);
        C2 v;
        return pair_corrects<R>(ev[p], ev[pj], a, v) ? v : mk<R>((R)0, (R)0);
      };
      top[b] = start(2 * t);
      bot[b] = start(2 * t + 1);
    }
    __syncthreads();  // the buffers are free
    bring(nchunk - 1, tid, THREADS);
    __syncthreads();
    for (int c = nchunk - 1; c >= 0; --c) {
      if (!col) {
        if (c > 0) bring(c - 1, tid - 32 * cw, THREADS - 32 * cw);
      } else {
        const Plane<R>* pl = (c & 1) ? buf1 : buf0;
        const int cnt = min(SR_CHUNK, K - c * SR_CHUNK);
        C2 ws[PPL];
        R wc[PPL];
#pragma unroll
        for (int b = 0; b < PPL; ++b) {
          const Plane<R> w = pl[(cnt - 1) * np + tp[b]];
          ws[b] = w.s;
          wc[b] = w.c;
        }
#pragma unroll 2
        for (int r = cnt - 1; r >= 0; --r) {
          // value that position p of this round has: the one at its next position
          const C2 below = mk<R>(__shfl_down_sync(0xffffffffu, top[0].x, 1, LANES),
                                 __shfl_down_sync(0xffffffffu, top[0].y, 1, LANES));
          const C2 above = mk<R>(__shfl_up_sync(0xffffffffu, bot[PPL - 1].x, 1, LANES),
                                 __shfl_up_sync(0xffffffffu, bot[PPL - 1].y, 1, LANES));
          C2 ns[PPL];  // the planes of the round before it, in flight meanwhile
          R nc[PPL];
          const Plane<R>* pn = pl + max(r - 1, 0) * np;
#pragma unroll
          for (int b = 0; b < PPL; ++b) {
            const Plane<R> w = pn[tp[b]];
            ns[b] = w.s;
            nc[b] = w.c;
          }
          C2 u[PPL], v[PPL];
#pragma unroll
          for (int b = 0; b < PPL; ++b) {
            u[b] = b + 1 < PPL ? top[b + 1 < PPL ? b + 1 : 0] : below;
            v[b] = b > 0 ? bot[b > 0 ? b - 1 : 0] : above;
            if (last[b]) u[b] = bot[b];
          }
          if (first) {
            v[0] = np == 1 ? bot[0] : u[0];
            u[0] = top[0];
          }
#pragma unroll
          for (int b = 0; b < PPL; ++b) {
            top[b] = zaxpy(wc[b], u[b], zmul(ws[b], v[b]));                               // c u + s v
            bot[b] = zaxpy(wc[b], v[b], zmul(mk<R>(-ws[b].x, ws[b].y), u[b]));            // c v - conj(s) u
            ws[b] = ns[b];
            wc[b] = nc[b];
          }
        }
      }
      __syncthreads();
    }
    if (col && j < ncols) {
#pragma unroll
      for (int b = 0; b < PPL; ++b) {
        const int p = 2 * (hl * PPL + b);
        if (p < nk_) Y[p * ldy + j] = top[b];
        if (p + 1 < nk_) Y[(p + 1) * ldy + j] = bot[b];
      }
    }
    c0 += PER * cw;
  }
  __syncthreads();
}

// The factor that makes nearly orthonormal columns X orthonormal in FP64: E = X^H X - I (n x n, row stride lde, and
// in FP32 in F, stride SR_LD) is replaced by M = I - E/2 + 3/8 E^2, the binomial series of (I + E)^-1/2; E^2 by
// FP32 products (their rounding stays below 1e-16 for the E let through).  Q = X M has Q^H Q - I = -5/8 E^3 to
// leading order.  Returns, to all threads, whether that is below FP64's rounding: ||E^3|| <= ||E^2||^1.5, and the row
// sums of |E^2|, which bound that norm, are held to 1e-10 (6e-16 is left).  Columns from rotations in FP32 have row sums of
// 2e-12 (n = 24) to 2.2e-11 (n = 72) at most on the reference solves' problems.
template <int THREADS>
__device__ __forceinline__ bool orthonormal_factor(const float2* F, double2* E, int lde, int n) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  bool bad = false;
  for (int i = warp; i < n; i += THREADS / 32) {
    float row = 0.f;
    for (int j = lane; j < n; j += 32) {
      float2 q = make_float2(0.f, 0.f);
      for (int p = 0; p < n; ++p) cfma(q, F[i * SR_LD + p], F[p * SR_LD + j]);
      row += fabsf(q.x) + fabsf(q.y);
      const double2 e = E[i * lde + j];
      E[i * lde + j] = make_double2((i == j ? 1.0 : 0.0) - 0.5 * e.x + 0.375 * q.x, -0.5 * e.y + 0.375 * q.y);
    }
    for (int o = 16; o > 0; o >>= 1) row += __shfl_xor_sync(0xffffffffu, row, o);
    bad |= !(row <= 1e-10f);  // also NaN
  }
  return !__syncthreads_or(bad);
}

// Conjugate-direction coefficients, inside the CTA that solved the projected problem.  With the
// Ritz coefficients cX (n x m, cX^H GO cX = I) of the basis S = [X_old, W, P_old], the next
// conjugate block spans the part of span(X_old) that is GO-orthogonal to the new Ritz block:
// Z = E - cX (cX^H GO E), E = [I_m; 0], projected once more, Z - cX (cX^H GO Z), and orthonormalised in
// the GO metric (H = Z^H GO Z, unit-diagonal scaled, Cholesky-QR; columns with H_jj at or below abs_drop
// are dropped), cP = Z T.  The second projection: once a column has nearly converged, Z is a difference
// of nearly equal vectors whose rounding lies in the Ritz block, and normalising it put noise at cosines
// of 0.5 to X into P, which broke single k-points of high-contrast cells late in the iteration (4 of 16
// start blocks on the SC 16^3 cell under the Young's-modulus law; none since).
// GO: the projected Gram matrix (global), of problem prob; G (stride SR_LD), cx, z, gz (n x m compact), Mm, Mi (m x m,
// stride m | 1), Dd (m), drp (m): shared workspaces; cp: output (n x m).  The products give each
// thread four rows of one column (the row operands are shared by the warp's lanes).
template <typename R, int THREADS, typename C2 = typename cplx_t<R>::type>
__device__ void pdir(const MatRef<R>& GO, int prob, int n, int m, R abs_drop, C2* G, const C2* cx, C2* z, C2* gz, C2* Mm, C2* Mi,
                     R* Dd, int* drp, C2* __restrict__ cp) {
  constexpr int W = THREADS / 32;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ldm = m | 1;
  for (int r = warp; r < n; r += W)  // GO, symmetrised
    for (int q = lane; q < n; q += 32) G[r * SR_LD + q] = GO.at(prob, r * n + q);
  __syncthreads();
  for (int r = warp; r < n; r += W)
    for (int q = r + lane; q < n; q += 32) {
      const C2 g1 = G[r * SR_LD + q], g2 = G[q * SR_LD + r];
      const C2 g = mk<R>((R)0.5 * (g1.x + g2.x), (R)0.5 * (g1.y - g2.y));
      G[r * SR_LD + q] = g;
      if (q > r) G[q * SR_LD + r] = cconj(g);
    }
  __syncthreads();
  const int mg = (m + 1) / 2, n4 = (n + 3) / 4;
  for (int t = tid; t < mg * m; t += THREADS) {  // M = cX^H GO E, two rows per thread
    const int g = t / m, j = t - g * m, i0 = 2 * g, i1 = min(2 * g + 1, m - 1);
    C2 s0 = mk<R>(0, 0), s1 = s0;
#pragma unroll 4
    for (int r = 0; r < n; ++r) {
      const C2 v = G[r * SR_LD + j];
      cfmac(s0, cx[r * m + i0], v);
      cfmac(s1, cx[r * m + i1], v);
    }
    Mm[i0 * ldm + j] = s0;
    if (2 * g + 1 < m) Mm[i1 * ldm + j] = s1;
  }
  __syncthreads();
  for (int t = tid; t < n4 * m; t += THREADS) {  // Z = E - cX M
    const int g = t / m, j = t - g * m;
    C2 s[4];
    int rr[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      rr[q] = min(4 * g + q, n - 1);
      s[q] = mk<R>(4 * g + q == j ? (R)1 : (R)0, (R)0);
    }
    for (int i = 0; i < m; ++i) {
      const C2 v = Mm[i * ldm + j];
#pragma unroll
      for (int q = 0; q < 4; ++q) cfma(s[q], zneg(cx[rr[q] * m + i]), v);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (4 * g + q < n) z[(4 * g + q) * m + j] = s[q];
  }
  __syncthreads();
  for (int t = tid; t < n4 * m; t += THREADS) {  // GZ = GO Z
    const int g = t / m, j = t - g * m;
    C2 s[4];
    int rr[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      rr[q] = min(4 * g + q, n - 1) * SR_LD;
      s[q] = mk<R>(0, 0);
    }
#pragma unroll 2
    for (int k = 0; k < n; ++k) {
      const C2 v = z[k * m + j];
#pragma unroll
      for (int q = 0; q < 4; ++q) cfma(s[q], G[rr[q] + k], v);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (4 * g + q < n) gz[(4 * g + q) * m + j] = s[q];
  }
  __syncthreads();
  // M2 = cX^H GZ and H = Z^H GZ, two rows per thread
  for (int t = tid; t < 2 * mg * m; t += THREADS) {
    const int w = t >= mg * m, u = t - w * mg * m;
    const int g = u / m, j = u - g * m, i0 = 2 * g, i1 = min(2 * g + 1, m - 1);
    const C2* left = w ? z : cx;
    C2* out = w ? Mi : Mm;
    C2 s0 = mk<R>(0, 0), s1 = s0;
#pragma unroll 4
    for (int r = 0; r < n; ++r) {
      const C2 v = gz[r * m + j];
      cfmac(s0, left[r * m + i0], v);
      cfmac(s1, left[r * m + i1], v);
    }
    out[i0 * ldm + j] = s0;
    if (2 * g + 1 < m) out[i1 * ldm + j] = s1;
  }
  __syncthreads();
  // Z <- Z - cX M2 (in place), and H <- H - M2^H M2 with it
  for (int t = tid; t < n4 * m; t += THREADS) {
    const int g = t / m, j = t - g * m;
    C2 s[4];
    int rr[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      rr[q] = min(4 * g + q, n - 1) * m;
      s[q] = z[rr[q] + j];
    }
    for (int i = 0; i < m; ++i) {
      const C2 v = Mm[i * ldm + j];
#pragma unroll
      for (int q = 0; q < 4; ++q) cfma(s[q], zneg(cx[rr[q] + i]), v);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (4 * g + q < n) z[rr[q] + j] = s[q];
  }
  for (int t = tid; t < m * m; t += THREADS) {
    const int i = t / m, j = t - i * m;
    C2 s = mk<R>(0, 0);
    for (int r = 0; r < m; ++r) cfmac(s, Mm[r * ldm + i], Mm[r * ldm + j]);
    Mi[i * ldm + j] = csub(Mi[i * ldm + j], s);
  }
  __syncthreads();
  if (tid < m) {  // column scales
    const R d = Mi[tid * ldm + tid].x;
    Dd[tid] = (d > abs_drop && d == d) ? (R)1 / sqrt(d) : (R)0;
    drp[tid] = 0;
  }
  __syncthreads();
  for (int t = tid; t < m * m; t += THREADS) {  // unit-diagonal scaled and symmetrised
    const int i = t / m, j = t - i * m;
    const C2 s1 = Mi[i * ldm + j], s2 = Mi[j * ldm + i];
    const R sc = Dd[i] * Dd[j] * (R)0.5;
    Mm[i * ldm + j] = mk<R>((s1.x + s2.x) * sc, (s1.y - s2.y) * sc);
  }
  __syncthreads();
  if (warp == 0) warp_chol_inverse<R>(Mm, Mi, m, ldm, (R)1e-10, drp);
  __syncthreads();
  for (int t = tid; t < n4 * m; t += THREADS) {  // cP = Z T, T[i][c] = D_i conj(Li[c][i]) for c >= i
    const int g = t / m, c = t - g * m;
    C2 s[4];
    int rr[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      rr[q] = min(4 * g + q, n - 1) * m;
      s[q] = mk<R>(0, 0);
    }
    if (!drp[c] && Dd[c] != (R)0) {
      for (int i = 0; i <= c; ++i) {
        const C2 li = Mi[c * ldm + i];
        const C2 v = mk<R>(li.x * Dd[i], -li.y * Dd[i]);
#pragma unroll
        for (int q = 0; q < 4; ++q) cfma(s[q], z[rr[q] + i], v);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (4 * g + q < n) cp[(4 * g + q) * m + c] = s[q];
  }
}

// Projected Rayleigh-Ritz problems of the FP32 block iteration: one CTA per k-point solves the
// Hermitian pencil (GA, GO) of the basis S = [X W P] (n <= 72 columns) for its lowest m
// eigenpairs, with eigenvalues accurate relative to their own size.
//
// Steps (per k):
//  1. unit-diagonal scaling D = diag(GO)^-1/2 and Hermitian symmetrisation of both matrices;
//  2. Cholesky GO = L L^H, blocked: the 8 x 8 diagonal block is factored in registers by the warps
//     that then solve the panel rows below it (one row per lane, shuffles instead of barriers);
//     the trailing update is shared by all warps.  A pivot at or below drop_tol drops its
//     coordinate (its row and column of L become e_j);
//  3. T = L^-1 GA and L^-1, then the upper triangle of C = L^-1 T^H = L^-1 GA L^-H, by right-looking
//     blocked forward substitution (8 x 8 diagonal solve, one thread per column, then the rank-8
//     update of the rows below, four rows per thread);
//  4. the kept coordinates are packed into a position-ordered upper-triangular copy of C and
//     diagonalised by cyclic two-sided Jacobi, the n_k/2 disjoint planes of a round ordered
//     by the circle method.  Positions are pair-ordered: the planes of every round are the
//     position pairs (2t, 2t+1), and the rotated matrix is written to the other buffer at the
//     positions the next round gives its indices.  So a thread reads and writes the same places in
//     every round (a full sweep is the identity permutation): its addresses and signs are computed
//     once, in registers, and a round is loads, rotations, stores and one barrier.  Warps have fixed
//     roles: 2 x 2 blocks of the matrix (one per thread) and the planes of the next round (three lanes
//     per plane, from the entries they need, recomputed with the same arithmetic as the block
//     updates).  The planes of every round are logged to global memory (L2).
//     A plane rotates when |a_uv| > eps sqrt(|a_uu a_vv|) + eps max_{i < m} |a_ii| (the absolute
//     floor is the rounding level of the current Ritz block); after each sweep one pass over the
//     pairs ends the iteration when none that concerns the m lowest would rotate.
//  5. the lowest m eigenvalues of the kept coordinates, their eigenvectors Y from the logged
//     rotations applied to m unit vectors, last round first, and the coefficients D L^-H Y;
//  6. when asked, the conjugate-direction coefficients of the next iteration from the same
//     CTA (pdir32: Cholesky-QR of the part of the old Ritz block outside the new one).
// Bound: the chain of a Jacobi round (barrier, plane loads, rotated entry, new plane: 740 of 970
// cycles at n = 57) for small n, issue and shared-memory bandwidth of one SM for n near 72.  50
// problems of the design workloads: n = 45 400 -> 177 us, n = 57 583 -> 279 us, n = 69 885 -> 389-437 us
// against positions that moved by index tables, V accumulated beside the rotations (its traffic was
// 60 % of the rounds' shared-memory bytes) and CTA-wide barriers in every column of the reductions.
// This is the mixed form's version (FP32, four 72 x 74 complex matrices in shared memory);
// the FP64 form keeps the kernel in lobpcg.cu.
#include "kernels.h"
#include "small_dense.cuh"

namespace {

constexpr int SR_THREADS = 1024;
constexpr int SR_NMAX = 72;
constexpr int SR_LD = 74;                       // even row stride: 16-byte aligned element pairs
constexpr int SR_MAT = SR_NMAX * SR_LD;         // complex elements per matrix
constexpr int SR_MAX_SWEEPS = 16;               // 5 to 7 are taken
constexpr int SR_PB = 8;                        // panel / row-block width of the reductions

// Complex arithmetic with explicit roundings, so that every call site computes bitwise the
// same value from the same inputs (the plane threads recompute entries the block threads
// store).
__device__ __forceinline__ float2 zmul(float2 a, float2 b) {
  return make_float2(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x)));
}
__device__ __forceinline__ float2 zconj(float2 a) { return make_float2(a.x, -a.y); }
// c x + z (c real)
__device__ __forceinline__ float2 zaxpy(float c, float2 x, float2 z) {
  return make_float2(__fmaf_rn(c, x.x, z.x), __fmaf_rn(c, x.y, z.y));
}
__device__ __forceinline__ float2 zneg(float2 a) { return make_float2(-a.x, -a.y); }

// Rotation of a plane: col_u <- c col_u - conj(s) col_v, col_v <- s col_u + c col_v; on: s != 0.
struct __align__(16) Plane {
  float2 s;
  float c;
  int on;
};

// Entry (r, col) of J1^H M J2 for a 2 x 2 block M (rows: plane 1, columns: plane 2) from the entries
// named relative to it: ms[a] = M[a == 0 ? r : 1 - r][col], mo[a] the same rows' other column.
// sg2 = -1 for col = 0, +1 for col = 1; sg1 the same of r.
__device__ __forceinline__ float2 rotated(float2 ms0, float2 mo0, float2 ms1, float2 mo1, const Plane& p1, float sg1,
                                          const Plane& p2, float sg2) {
  const float2 s2 = make_float2(sg2 * p2.s.x, p2.s.y);    // -conj(s) or s
  const float2 y0 = zaxpy(p2.c, ms0, zmul(s2, mo0)), y1 = zaxpy(p2.c, ms1, zmul(s2, mo1));
  const float2 s1 = make_float2(sg1 * p1.s.x, -p1.s.y);   // -s or conj(s)
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
__device__ __forceinline__ Plane make_plane(float app, float aqq, float2 apq, float floor_abs) {
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
  Plane w;
  w.c = on ? c : 1.f;
  w.s = make_float2(on ? f * apq.x : 0.f, on ? f * apq.y : 0.f);
  w.on = on ? 1 : 0;
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
__device__ __forceinline__ void block_cholesky(float2* B, int n, float drop_tol, int* drop, float* invd) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int j0 = 0; j0 < n; j0 += SR_PB) {
    const int jb = min(SR_PB, n - j0), j1 = j0 + jb;
    float2 a[SR_PB];
    if (warp == 0 || j1 + 32 * warp < n) {
      // every warp with panel rows factors the diagonal block (row lane % 8) for itself
      const int r = lane & 7;
      float inv[SR_PB];
#pragma unroll
      for (int c = 0; c < SR_PB; ++c) a[c] = (r < jb && c < jb) ? B[(j0 + r) * SR_LD + j0 + c] : make_float2(0.f, 0.f);
#pragma unroll
      for (int j = 0; j < SR_PB; ++j) {
        const float d = __shfl_sync(0xffffffffu, a[j].x, j);
        const bool keep = d > drop_tol;
        const float sq = sqrtf(d);
        inv[j] = keep ? 1.f / sq : 0.f;
        if (r == j) a[j] = make_float2(keep ? sq : 1.f, 0.f);
        else a[j] = make_float2(a[j].x * inv[j], a[j].y * inv[j]);
#pragma unroll
        for (int c = j + 1; c < SR_PB; ++c) {
          const float2 lc = make_float2(__shfl_sync(0xffffffffu, a[j].x, c), __shfl_sync(0xffffffffu, a[j].y, c));
          if (r >= c) {  // a_rc -= l_rj conj(l_cj)
            a[c].x -= a[j].x * lc.x + a[j].y * lc.y;
            a[c].y -= a[j].y * lc.x - a[j].x * lc.y;
          }
        }
      }
      const int i = j1 + 32 * warp + lane;
      float2 b[SR_PB];
#pragma unroll
      for (int c = 0; c < SR_PB; ++c) b[c] = i < n && c < jb ? B[i * SR_LD + j0 + c] : make_float2(0.f, 0.f);
#pragma unroll
      for (int j = 0; j < SR_PB; ++j) {
#pragma unroll
        for (int k = 0; k < j; ++k) {
          const float2 l = make_float2(__shfl_sync(0xffffffffu, a[k].x, j), __shfl_sync(0xffffffffu, a[k].y, j));
          b[j].x -= b[k].x * l.x + b[k].y * l.y;
          b[j].y -= b[k].y * l.x - b[k].x * l.y;
        }
        b[j].x *= inv[j];
        b[j].y *= inv[j];
      }
      if (i < n)
#pragma unroll
        for (int c = 0; c < SR_PB; ++c)
          if (c < jb) B[i * SR_LD + j0 + c] = b[c];
      if (warp == 0)
#pragma unroll
        for (int c = 0; c < SR_PB; ++c)
          if (lane == c && c < jb) {
            drop[j0 + c] = inv[c] == 0.f ? 1 : 0;
            invd[j0 + c] = inv[c] == 0.f ? 1.f : inv[c];
          }
    }
    __syncthreads();
    if (warp == 0 && lane < jb)  // every warp has read the diagonal block
#pragma unroll
      for (int c = 0; c < SR_PB; ++c)
        if (c <= lane) B[(j0 + lane) * SR_LD + j0 + c] = a[c];
    // trailing update of the rows and columns from j1 on by the panel (dropped columns are zero)
    const int nt = n - j1;
    for (int rr = warp; rr < nt; rr += 32) {
      const int i = j1 + rr;
      const float4* Li = reinterpret_cast<const float4*>(B + i * SR_LD + j0);
      for (int q = lane; q <= rr; q += 32) {
        const int c = j1 + q;
        const float4* Lc = reinterpret_cast<const float4*>(B + c * SR_LD + j0);
        float2 v = B[i * SR_LD + c];
#pragma unroll
        for (int h = 0; h < SR_PB / 2; ++h) {  // jb = SR_PB wherever rows remain below the panel
          const float4 x = Li[h], y = Lc[h];
          v.x -= x.x * y.x + x.y * y.y;
          v.y -= x.y * y.x - x.x * y.y;
          v.x -= x.z * y.z + x.w * y.w;
          v.y -= x.w * y.z - x.z * y.w;
        }
        B[i * SR_LD + c] = v;
      }
    }
    __syncthreads();
  }
  for (int i = warp; i < n; i += 32)
    for (int c = lane; c <= i; c += 32)
      if (drop[i] || drop[c]) B[i * SR_LD + c] = make_float2(i == c ? 1.f : 0.f, 0.f);
  __syncthreads();
}

// Forward substitution L X = R in place, right-looking in blocks of 8 rows.  Columns c < n0 of R are
// columns of P0, the others columns c - n0 of P1.  tri = 1: P1 starts as the identity, whose
// column j is zero above row j; tri = 2 (n0 = ncol): only rows i <= c of column c are wanted.
__device__ __forceinline__ void block_forward(const float2* L, const float* invd, float2* P0, float2* P1, int n0, int n,
                                              int ncol, int tri) {
  const int tid = threadIdx.x;
  for (int i0 = 0; i0 < n; i0 += SR_PB) {
    const int ib = min(SR_PB, n - i0), i1 = i0 + ib;
    const int c_lo = tri == 2 ? i0 : 0;
    const int c_hi = tri == 1 ? n0 + min(n, i1) : ncol;
    for (int c = c_lo + tid; c < c_hi; c += SR_THREADS) {
      float2* R = c < n0 ? P0 + c : P1 + (c - n0);
      float2 x[SR_PB];
#pragma unroll
      for (int ii = 0; ii < SR_PB; ++ii) {
        if (ii < ib) {
          const int i = i0 + ii;
          float2 acc = R[i * SR_LD];
#pragma unroll
          for (int kk = 0; kk < ii; ++kk) {
            const float2 l = L[i * SR_LD + i0 + kk];
            acc.x -= l.x * x[kk].x - l.y * x[kk].y;
            acc.y -= l.x * x[kk].y + l.y * x[kk].x;
          }
          x[ii] = make_float2(acc.x * invd[i], acc.y * invd[i]);
          R[i * SR_LD] = x[ii];
        }
      }
    }
    __syncthreads();
    if (i1 >= n) break;
    // rows below: four rows of one column per thread (i1 is a multiple of 8 here)
    const int nc = c_hi - c_lo, ng = (n - i1 + 3) / 4;
    for (int e = tid; e < nc * ng; e += SR_THREADS) {
      const int g = e / nc, c = c_lo + e - g * nc;
      const int r0 = i1 + 4 * g;
      if (tri == 2 && c < r0) continue;
      float2* R = c < n0 ? P0 + c : P1 + (c - n0);
      float2 acc[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] = make_float2(0.f, 0.f);
#pragma unroll
      for (int k = 0; k < SR_PB; ++k) {
        const float2 x = R[(i0 + k) * SR_LD];
#pragma unroll
        for (int q = 0; q < 4; ++q) cfma(acc[q], L[(r0 + q) * SR_LD + i0 + k], x);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (r0 + q < n) R[(r0 + q) * SR_LD] = csub(R[(r0 + q) * SR_LD], acc[q]);
    }
    __syncthreads();
  }
}

__device__ __forceinline__ float4 as_float4(const Plane& w) {
  return make_float4(w.s.x, w.s.y, w.c, __int_as_float(w.on));
}

// Eigenvectors of the packed matrix from the logged rotations (np planes per round, K rounds):
// column j of Y (nk_ x m) = J_1 P_1 J_2 P_2 ... J_K P_K e, e the unit vector of position perm[j],
// P the circle method's moves.  Applied to the m wanted columns only, from the last round back, which
// is a third of the work of accumulating all of V beside the rotations and leaves the shared-memory
// bandwidth of the rounds to the matrix (it was their bound: 147 KB a round at n = 69, of which
// V took 87).  Half a warp holds a column, PPL planes (2 PPL positions) per lane in registers; a move
// is one complex value from each neighbouring lane.  The other warps bring the log from L2 in chunks
// of SR_CHUNK rounds, one ahead.
constexpr int SR_CHUNK = 64;  // rounds x 36 planes x 16 bytes = 36 KB per buffer
template <int PPL>
__device__ __forceinline__ void replay(const float4* __restrict__ logk, int K, int np, int nk_, int m, const int* perm,
                                       float4* buf0, float4* buf1, float2* Y) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cw = (m + 1) / 2;  // warps that hold columns
  const int hl = lane & 15, j = 2 * warp + (lane >> 4);
  const bool col = warp < cw;
  float2 top[PPL], bot[PPL];
  int tp[PPL];       // plane read (those past the last hold nothing: their values reach no column)
  bool last[PPL];
  const bool first = hl == 0;
#pragma unroll
  for (int b = 0; b < PPL; ++b) {
    tp[b] = min(hl * PPL + b, np - 1);
    last[b] = hl * PPL + b == np - 1;
  }
  if (col) {
    const int p = j < m ? perm[j] : -1;
#pragma unroll
    for (int b = 0; b < PPL; ++b) {
      const int t = hl * PPL + b;
      top[b] = make_float2(2 * t == p ? 1.f : 0.f, 0.f);
      bot[b] = make_float2(2 * t + 1 == p ? 1.f : 0.f, 0.f);
    }
  }
  const int nchunk = (K + SR_CHUNK - 1) / SR_CHUNK;
  auto bring = [&](int c, int first, int step) {  // rounds c SR_CHUNK .. of the log
    float4* dst = (c & 1) ? buf1 : buf0;
    const int cnt = min(SR_CHUNK, K - c * SR_CHUNK) * np;
    const float4* src = logk + (long long)c * SR_CHUNK * np;
    for (int e = first; e < cnt; e += step) dst[e] = __ldcg(src + e);
  };
  __syncthreads();  // the buffers are free
  bring(nchunk - 1, tid, SR_THREADS);
  __syncthreads();
  for (int c = nchunk - 1; c >= 0; --c) {
    if (!col) {
      if (c > 0) bring(c - 1, tid - 32 * cw, SR_THREADS - 32 * cw);
    } else {
      const float4* pl = ((c & 1) ? buf1 : buf0);
      const int cnt = min(SR_CHUNK, K - c * SR_CHUNK);
      float4 w[PPL];
#pragma unroll
      for (int b = 0; b < PPL; ++b) w[b] = pl[(cnt - 1) * np + tp[b]];
#pragma unroll 2
      for (int r = cnt - 1; r >= 0; --r) {
        // value that position p of this round has: the one at its next position
        const float2 below = make_float2(__shfl_down_sync(0xffffffffu, top[0].x, 1, 16),
                                         __shfl_down_sync(0xffffffffu, top[0].y, 1, 16));
        const float2 above = make_float2(__shfl_up_sync(0xffffffffu, bot[PPL - 1].x, 1, 16),
                                         __shfl_up_sync(0xffffffffu, bot[PPL - 1].y, 1, 16));
        float4 nw[PPL];  // the planes of the round before it, in flight meanwhile
        const float4* pn = pl + max(r - 1, 0) * np;
#pragma unroll
        for (int b = 0; b < PPL; ++b) nw[b] = pn[tp[b]];
        float2 u[PPL], v[PPL];
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
          const float2 s = make_float2(w[b].x, w[b].y);
          top[b] = zaxpy(w[b].z, u[b], zmul(s, v[b]));                           // c u + s v
          bot[b] = zaxpy(w[b].z, v[b], zmul(make_float2(-s.x, s.y), u[b]));      // c v - conj(s) u
          w[b] = nw[b];
        }
      }
    }
    __syncthreads();
  }
  if (col && j < m) {
#pragma unroll
    for (int b = 0; b < PPL; ++b) {
      const int p = 2 * (hl * PPL + b);
      if (p < nk_) Y[p * m + j] = top[b];
      if (p + 1 < nk_) Y[(p + 1) * m + j] = bot[b];
    }
  }
  __syncthreads();
}

// Conjugate-direction coefficients, inside the CTA that solved the projected problem.  With the
// Ritz coefficients cX (n x m, cX^H GO cX = I) of the basis S = [X_old, W, P_old], the next
// conjugate block spans the part of span(X_old) that is GO-orthogonal to the new Ritz block:
// Z = E - cX (cX^H GO E), E = [I_m; 0], orthonormalised in the GO metric (H = Z^H GO Z,
// unit-diagonal scaled, Cholesky-QR; columns with H_jj at or below abs_drop carry only rounding
// and are dropped), cP = Z T.  go: the projected Gram matrix (global); G (stride SR_LD), cx, z, gz
// (n x m compact), Mm (m x m), tmp (m), Dd (m), drp (m): shared workspaces; cp: output (n x m).
// go: the projected Gram matrix (global); G (stride SR_LD), cx, z, gz (n x m compact), Mm, Mi (m x m,
// stride m | 1), Dd (m), drp (m): shared workspaces; cp: output (n x m).  The products give each
// thread four rows of one column (the row operands are shared by the warp's lanes).
__device__ void pdir32(const float2* __restrict__ go, int n, int m, float abs_drop, float2* G, const float2* cx,
                       float2* z, float2* gz, float2* Mm, float2* Mi, float* Dd, int* drp, float2* __restrict__ cp) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ldm = m | 1;
  for (int r = warp; r < n; r += 32)  // GO, symmetrised
    for (int q = lane; q < n; q += 32) {
      const float2 g1 = go[r * n + q], g2 = go[q * n + r];
      G[r * SR_LD + q] = make_float2(0.5f * (g1.x + g2.x), 0.5f * (g1.y - g2.y));
    }
  __syncthreads();
  const int mg = (m + 1) / 2, n4 = (n + 3) / 4;
  for (int t = tid; t < mg * m; t += SR_THREADS) {  // M = cX^H GO E, two rows per thread
    const int g = t / m, j = t - g * m, i0 = 2 * g, i1 = min(2 * g + 1, m - 1);
    float2 s0 = make_float2(0.f, 0.f), s1 = s0;
#pragma unroll 4
    for (int r = 0; r < n; ++r) {
      const float2 v = G[r * SR_LD + j];
      cfmac(s0, cx[r * m + i0], v);
      cfmac(s1, cx[r * m + i1], v);
    }
    Mm[i0 * ldm + j] = s0;
    if (2 * g + 1 < m) Mm[i1 * ldm + j] = s1;
  }
  __syncthreads();
  for (int t = tid; t < n4 * m; t += SR_THREADS) {  // Z = E - cX M
    const int g = t / m, j = t - g * m;
    float2 s[4];
    int rr[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      rr[q] = min(4 * g + q, n - 1);
      s[q] = make_float2(4 * g + q == j ? 1.f : 0.f, 0.f);
    }
    for (int i = 0; i < m; ++i) {
      const float2 v = Mm[i * ldm + j];
#pragma unroll
      for (int q = 0; q < 4; ++q) cfma(s[q], zneg(cx[rr[q] * m + i]), v);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (4 * g + q < n) z[(4 * g + q) * m + j] = s[q];
  }
  __syncthreads();
  for (int t = tid; t < n4 * m; t += SR_THREADS) {  // GZ = GO Z
    const int g = t / m, j = t - g * m;
    float2 s[4];
    int rr[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      rr[q] = min(4 * g + q, n - 1) * SR_LD;
      s[q] = make_float2(0.f, 0.f);
    }
#pragma unroll 2
    for (int k = 0; k < n; ++k) {
      const float2 v = z[k * m + j];
#pragma unroll
      for (int q = 0; q < 4; ++q) cfma(s[q], G[rr[q] + k], v);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (4 * g + q < n) gz[(4 * g + q) * m + j] = s[q];
  }
  __syncthreads();
  for (int t = tid; t < mg * m; t += SR_THREADS) {  // H = Z^H GZ, two rows per thread
    const int g = t / m, j = t - g * m, i0 = 2 * g, i1 = min(2 * g + 1, m - 1);
    float2 s0 = make_float2(0.f, 0.f), s1 = s0;
#pragma unroll 4
    for (int r = 0; r < n; ++r) {
      const float2 v = gz[r * m + j];
      cfmac(s0, z[r * m + i0], v);
      cfmac(s1, z[r * m + i1], v);
    }
    Mi[i0 * ldm + j] = s0;
    if (2 * g + 1 < m) Mi[i1 * ldm + j] = s1;
  }
  __syncthreads();
  if (tid < m) {  // column scales
    const float d = Mi[tid * ldm + tid].x;
    Dd[tid] = (d > abs_drop && d == d) ? 1.f / sqrtf(d) : 0.f;
    drp[tid] = 0;
  }
  __syncthreads();
  for (int t = tid; t < m * m; t += SR_THREADS) {  // unit-diagonal scaled and symmetrised
    const int i = t / m, j = t - i * m;
    const float2 s1 = Mi[i * ldm + j], s2 = Mi[j * ldm + i];
    const float sc = Dd[i] * Dd[j] * 0.5f;
    Mm[i * ldm + j] = make_float2((s1.x + s2.x) * sc, (s1.y - s2.y) * sc);
  }
  __syncthreads();
  if (warp == 0) warp_chol_inverse<float>(Mm, Mi, m, ldm, 1e-10f, drp);
  __syncthreads();
  for (int t = tid; t < n4 * m; t += SR_THREADS) {  // cP = Z T, T[i][c] = D_i conj(Li[c][i]) for c >= i
    const int g = t / m, c = t - g * m;
    float2 s[4];
    int rr[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      rr[q] = min(4 * g + q, n - 1) * m;
      s[q] = make_float2(0.f, 0.f);
    }
    if (!drp[c] && Dd[c] != 0.f) {
      for (int i = 0; i <= c; ++i) {
        const float2 li = Mi[c * ldm + i];
        const float2 v = make_float2(li.x * Dd[i], -li.y * Dd[i]);
#pragma unroll
        for (int q = 0; q < 4; ++q) cfma(s[q], z[rr[q] + i], v);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (4 * g + q < n) cp[(4 * g + q) * m + c] = s[q];
  }
}

}  // namespace

__global__ __launch_bounds__(SR_THREADS) void k_small_rr32(const float2* __restrict__ GA, const float2* __restrict__ GO,
                                                         int n, int m, float drop_tol, const int* __restrict__ kdone,
                                                         float* __restrict__ lam_out, float2* __restrict__ coef,
                                                         float2* __restrict__ cpo, float pdir_abs, int* status,
                                                         double* flops, float4* __restrict__ rotlog, long long log_stride) {
  extern __shared__ __align__(16) unsigned char smem[];
  float2* B0 = (float2*)smem;          // GO -> L -> Jacobi buffer 1
  float2* B1 = B0 + SR_MAT;            // GA -> T = L^-1 GA -> Jacobi buffer 0
  float2* Vt = B1 + SR_MAT;            // L^-1
  float2* Cm = Vt + SR_MAT;            // C = L^-1 GA L^-H (original order) -> Y
  Plane* pl = (Plane*)(Cm + SR_MAT);   // 2 x 36 planes (by round parity)
  float* D = (float*)(pl + 2 * 36);    // SR_NMAX
  float* ev = D + SR_NMAX;             // SR_NMAX: reciprocal diagonal of L, then eigenvalues
  int* drop = (int*)(ev + SR_NMAX);    // SR_NMAX
  int* idx = drop + SR_NMAX;           // SR_NMAX: position -> coordinate (-1: padding)
  int* perm = idx + SR_NMAX;           // SR_NMAX
  int* low = perm + SR_NMAX;           // SR_NMAX: among the m smallest diagonal entries
  int* misc = low + SR_NMAX;           // [0] kept count, [2] floor bits, [3] sweeps
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int k = blockIdx.x;
  const float2* ga = GA + (long long)k * n * n;
  const float2* go = GO + (long long)k * n * n;
  float4* logk = rotlog + k * log_stride;  // rotations of this problem, np planes per round
  float2* ck = coef + (long long)k * n * m;
  float2* cpk = cpo ? cpo + (long long)k * n * m : nullptr;  // conjugate-direction coefficients (or none)
  if (kdone && kdone[k]) {  // locked k-point: keep its block, leave lambda untouched, no conjugate block
    for (int t = tid; t < n * m; t += blockDim.x) {
      const int i = t / m, j = t % m;
      ck[t] = make_float2(i == j ? 1.f : 0.f, 0.f);
      if (cpk) cpk[t] = make_float2(0.f, 0.f);
    }
    return;
  }
  // 1. scaling, symmetrised copies, identity right-hand side of L^-1 (in Vt)
  for (int i = tid; i < n; i += blockDim.x) {
    const float d = go[i * n + i].x;
    D[i] = (d > 0.f && d == d) ? 1.f / sqrtf(d) : 0.f;
    drop[i] = 0;
  }
  __syncthreads();
  for (int i = warp; i < n; i += 32)
    for (int c = lane; c < n; c += 32) {
      const float2 a1 = ga[i * n + c], a2 = ga[c * n + i];
      const float2 b1 = go[i * n + c], b2 = go[c * n + i];
      const float s = D[i] * D[c] * 0.5f;
      B1[i * SR_LD + c] = make_float2((a1.x + a2.x) * s, (a1.y - a2.y) * s);
      B0[i * SR_LD + c] = make_float2((b1.x + b2.x) * s, (b1.y - b2.y) * s);
      Vt[i * SR_LD + c] = make_float2(i == c ? 1.f : 0.f, 0.f);
    }
  __syncthreads();
  // 2. Cholesky of B0 (lower)
  block_cholesky(B0, n, drop_tol, drop, ev);
  // 3. T = L^-1 GA (in place in B1) and L^-1 (in place in Vt), then C = L^-1 T^H in Cm (upper)
  block_forward(B0, ev, B1, Vt, n, n, 2 * n, 1);
  for (int i = warp; i < n; i += 32)
    for (int j = lane; j < n; j += 32) Cm[i * SR_LD + j] = zconj(B1[j * SR_LD + i]);
  __syncthreads();
  block_forward(B0, ev, Cm, nullptr, n, n, n, 2);
  if (tid == 0) {
    int kept = 0;
    for (int i = 0; i < n; ++i)
      if (!drop[i]) idx[kept++] = i;
    misc[0] = kept;
    if (kept & 1) idx[kept] = -1;  // padding position
  }
  __syncthreads();
  const int nk_ = misc[0];
  if (nk_ < m) {
    // too few independent directions: keep the current block (identity on its first m coordinates)
    for (int t = tid; t < n * m; t += blockDim.x) {
      const int i = t / m, j = t % m;
      ck[t] = make_float2(i == j ? 1.f : 0.f, 0.f);
    }
    for (int j = tid; j < m; j += blockDim.x) lam_out[(long long)k * m + j] = ga[j * n + j].x / go[j * n + j].x;
    if (tid == 0) set_status(status, PC_ENOCONV);
    if (cpk) {
      for (int t = tid; t < n * m; t += blockDim.x) {
        const int i = t / m, j = t % m;
        B1[t] = make_float2(i == j ? 1.f : 0.f, 0.f);
      }
      __syncthreads();
      pdir32(go, n, m, pdir_abs, B0, B1, B1 + n * m, B1 + 2 * n * m, Cm, Cm + m * (m | 1), ev, drop, cpk);
    }
    return;
  }
  const int npad = nk_ + (nk_ & 1), np = npad / 2, nrounds = npad - 1;
  const int nblk = np * (np + 1) / 2;
  // 4. packed position-ordered upper copy in B1 (T is no longer needed)
  for (int i = warp; i < npad; i += 32)
    for (int j = i + lane; j < npad; j += 32) {
      const int a = idx[i], b = idx[j];
      float2 v = (a < 0 || b < 0) ? make_float2(0.f, 0.f) : Cm[a * SR_LD + b];
      if (i == j) v.y = 0.f;
      B1[spos(i, j)] = v;
    }
  __syncthreads();
  // rounding floor: eps * max |a_ii| over the kept coordinates of the current Ritz block
  if (warp == 0) {
    float mx = 0.f;
    for (int p = lane; p < nk_; p += 32)
      if (idx[p] < m) mx = fmaxf(mx, fabsf(B1[spos(p, p)].x));
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) misc[2] = __float_as_int(1.1920929e-07f * mx);
  }
  __syncthreads();
  const float floor_abs = __int_as_float(misc[2]);
  if (tid < np) {  // planes of the first round
    const int u = 2 * tid, v = u + 1;
    const Plane w = make_plane(B1[spos(u, u)].x, B1[spos(v, v)].x, B1[spos(u, v)], floor_abs);
    pl[tid] = w;
    logk[tid] = as_float4(w);
  }
  __syncthreads();
  // Jacobi sweeps.  Roles by warp, in this order: pw plane warps (ten planes of three lanes each) and
  // bw block warps (one 2 x 2 block of the upper triangle per thread).  Only these take part in the
  // rounds' barriers; the rest wait at the end.  S is in B1 in even rounds and B0 in odd ones.
  const int pw = (np + 9) / 10, bw = (nblk + 31) / 32;
  const int nact = 32 * (pw + bw);
  int sweeps = 0, par = 0;
  // After a sweep every index is back at its own position.  Only the m lowest eigenpairs are wanted:
  // converged when no pair with one of the m smallest diagonal entries would rotate and the other
  // pairs are below 1e-3 of sqrt(a_ii a_jj), which keeps the eigenvalues among them away from the
  // lowest (each within 7 % of a diagonal entry for n <= 72).  Saves the last sweep of about half the
  // problems against asking it of all pairs.  ev: the diagonal, perm: positions by ascending entry.
  auto more = [&]() {
    ++sweeps;
    const float2* S = par ? B0 : B1;
    for (int p = tid; p < nk_; p += nact) ev[p] = S[spos(p, p)].x;
    bar_first(nact);
    for (int p = tid; p < nk_; p += nact) {
      int r = 0;
      const float vi = ev[p];
      for (int q = 0; q < nk_; ++q) r += (ev[q] < vi || (ev[q] == vi && q < p)) ? 1 : 0;
      perm[r] = p;
      low[p] = r < m ? 1 : 0;
    }
    bar_first(nact);
    bool any = false;
    for (int i = warp; i < nk_; i += nact / 32) {
      const float aii = ev[i];
      const int li = low[i];
      for (int j = i + 1 + lane; j < nk_; j += 32) {
        const float2 a = S[spos(i, j)];
        const float b2 = __fmaf_rn(a.x, a.x, a.y * a.y);
        any |= (li | low[j]) ? plane_rotates(aii, ev[j], b2, floor_abs) : b2 > 1e-6f * fabsf(aii * ev[j]) + floor_abs * floor_abs;
      }
    }
    return bar_first_or(nact, any) && sweeps < SR_MAX_SWEEPS;
  };
  auto flip = [](float2 a, unsigned f) { return make_float2(a.x, __uint_as_float(__float_as_uint(a.y) ^ f)); };
  if (warp < pw) {
    // plane pt of the next round from the entries at its positions u0, v0 of this one:
    // pe = 0: a_uu, 1: a_vv, 2: a_uv
    const int pt = warp * 10 + lane / 3, pe = lane % 3, pbase = lane - pe;
    const bool mine = lane < 30 && pt < np;
    int l0 = 0, l1 = 0, l2 = 0, l3 = 0, t1 = 0, t2 = 0;
    unsigned g0 = 0, g1 = 0, g2 = 0, g3 = 0, ge = 0;
    float sg1 = 0.f, sg2 = 0.f;
    if (mine) {
      const int u0 = prev_pos(2 * pt, np), v0 = prev_pos(2 * pt + 1, np);
      int u = pe == 1 ? v0 : u0, v = pe == 0 ? u0 : v0;
      if ((u >> 1) > (v >> 1)) {  // the stored block is the transposed one: conjugate the result
        const int x = u;
        u = v;
        v = x;
        ge = 0x80000000u;
      }
      t1 = u >> 1;
      t2 = v >> 1;
      const int r = u & 1, c = v & 1;
      sg1 = r ? 1.f : -1.f;
      sg2 = c ? 1.f : -1.f;
      // entries M[r][c], M[r][1-c], M[1-r][c], M[1-r][1-c]; below the diagonal the conjugate above it
      auto at = [&](int rr, int cc, unsigned& f) {
        const int i = 2 * t1 + rr, j = 2 * t2 + cc;
        if (i > j) f = 0x80000000u;
        return i <= j ? spos(i, j) : spos(j, i);
      };
      l0 = at(r, c, g0);
      l1 = at(r, 1 - c, g1);
      l2 = at(1 - r, c, g2);
      l3 = at(1 - r, 1 - c, g3);
    }
    float4* log_next = logk + np;
    do {
      for (int round = 0; round < nrounds; ++round) {
        const float2* S = par ? B0 : B1;
        const Plane* cur = pl + par * 36;
        const Plane p1 = cur[t1], p2 = cur[t2];
        float2 e = rotated(flip(S[l0], g0), flip(S[l1], g1), flip(S[l2], g2), flip(S[l3], g3), p1, sg1, p2, sg2);
        if (np == 1 && p1.on) e = make_float2(pe == 2 ? 0.f : e.x, 0.f);  // its own plane annihilated it
        e = flip(e, ge);
        const float auu = __shfl_sync(0xffffffffu, e.x, pbase & 31);
        const float avv = __shfl_sync(0xffffffffu, e.x, (pbase + 1) & 31);
        const float2 auv = make_float2(__shfl_sync(0xffffffffu, e.x, (pbase + 2) & 31),
                                       __shfl_sync(0xffffffffu, e.y, (pbase + 2) & 31));
        if (mine && pe == 0) {
          const Plane w = make_plane(auu, avv, auv, floor_abs);
          pl[(par ^ 1) * 36 + pt] = w;
          log_next[pt] = as_float4(w);
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
    unsigned f0 = 0, f1 = 0, f2 = 0, f3 = 0;
    if (mine) {
      int rem = u;
      while (rem >= np - t1) { rem -= np - t1; ++t1; }
      t2 = t1 + rem;
      l0 = spos(2 * t1, 2 * t2);
      const int ra = next_pos(2 * t1, np), rb = next_pos(2 * t1 + 1, np);
      const int ca = next_pos(2 * t2, np), cb = next_pos(2 * t2 + 1, np);
      auto to = [&](int i, int j, unsigned& f) {
        if (i > j) f = 0x80000000u;
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
          const float2* S = par ? B0 : B1;
          float2* T = par ? B1 : B0;
          const Plane* cur = pl + par * 36;
          const Plane p1 = cur[t1], p2 = cur[t2];
          const float2 m00 = S[l0], m01 = S[l0 + SR_LD / 2], m11 = S[l0 + SR_LD + SR_LD / 2];
          float2 m10 = S[l0 + SR_LD];
          if (dg) m10 = zconj(m01);
          float2 e00 = rotated(m00, m01, m10, m11, p1, -1.f, p2, -1.f);
          float2 e01 = rotated(m01, m00, m11, m10, p1, -1.f, p2, 1.f);
          const float2 e10 = rotated(m10, m11, m00, m01, p1, 1.f, p2, -1.f);
          float2 e11 = rotated(m11, m10, m01, m00, p1, 1.f, p2, 1.f);
          if (dg) {
            e00.y = 0.f;
            e11.y = 0.f;
            if (p1.on) e01 = make_float2(0.f, 0.f);
          } else {
            T[w2] = flip(e10, f2);
          }
          T[w0] = flip(e00, f0);
          T[w1] = flip(e01, f1);
          T[w3] = flip(e11, f3);
        }
        bar_first(nact);
        par ^= 1;
      }
    } while (more());
  }
  __syncthreads();
  // 5. lowest m eigenpairs of the kept coordinates
  sweeps = misc[3];
  // eigenvectors of the packed matrix for these m: the logged rotations, last round first
  float2* Y = Cm;  // nk_ x m
  const int K = sweeps * nrounds;
  if (np <= 16) replay<1>(logk, K, np, nk_, m, perm, (float4*)B1, (float4*)B0, Y);
  else if (np <= 32) replay<2>(logk, K, np, nk_, m, perm, (float4*)B1, (float4*)B0, Y);
  else replay<3>(logk, K, np, nk_, m, perm, (float4*)B1, (float4*)B0, Y);
  // coefficients D L^-H Y
  const int n4 = (n + 3) / 4;
  for (int t = tid; t < n4 * m; t += SR_THREADS) {
    const int g = t / m, j = t - g * m;
    float2 a[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int p = 0; p < nk_; ++p) {
      const float2 y = Y[p * m + j];
      const float2* li = Vt + idx[p] * SR_LD + 4 * g;  // columns past n: unused sums
#pragma unroll
      for (int q = 0; q < 4; ++q) cfmac(a[q], li[q], y);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = 4 * g + q;
      if (i < n) {
        const float2 c = make_float2(a[q].x * D[i], a[q].y * D[i]);
        ck[i * m + j] = c;
        B1[i * m + j] = c;  // cX for the conjugate directions
      }
    }
  }
  for (int j = tid; j < m; j += blockDim.x) lam_out[(long long)k * m + j] = ev[perm[j]];
  if (cpk) {
    __syncthreads();
    pdir32(go, n, m, pdir_abs, B0, B1, B1 + n * m, B1 + 2 * n * m, Cm, Cm + m * (m | 1), ev, drop, cpk);
  }
  if (flops && tid == 0) {
    // algorithmic work: Cholesky n^3/6, L^-1 GA n^3/2, L^-1 T^H n^3/2 and L^-1 n^3/6 complex
    // multiply-adds (8 real flops each); per Jacobi sweep n_k (n_k - 1) / 2 rotations, each
    // updating 2 n_k entries of C and 2 n entries of V at 12 real flops per entry
    const double nn = n, kk = nk_;
    atomicAdd(flops, 8.0 * (4.0 / 3.0) * nn * nn * nn + sweeps * kk * (kk - 1.0) * 0.5 * 24.0 * (kk + nn));
  }
}

// Rotations of the most sweeps, and the planes of the round after them.
long long small_rr32_log(int n) { return ((long long)SR_MAX_SWEEPS * n + 1) * ((n + 1) / 2); }

int launch_small_rr32(const float2* GA, const float2* GO, int n, int m, int nk, float drop_tol, const int* kdone,
                      float* lam_out, float2* coef, float2* cp, float pdir_abs, int* status, double* flops,
                      float4* rotlog, long long log_stride, cudaStream_t s) {
  if (n > SR_NMAX || m > n || n < 1 || log_stride < small_rr32_log(n)) return PC_EINVAL;
  const size_t sm = sizeof(float2) * 4 * (size_t)SR_MAT + sizeof(Plane) * 72 + sizeof(float) * 2 * SR_NMAX +
                    sizeof(int) * (4 * SR_NMAX + 8);
  static const cudaError_t attr =  // once, thread-safe (k groups launch from several host threads)
      cudaFuncSetAttribute(k_small_rr32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  (void)attr;
  k_small_rr32<<<nk, SR_THREADS, sm, s>>>(GA, GO, n, m, drop_tol, kdone, lam_out, coef, cp, pdir_abs, status, flops, rotlog,
                                             log_stride);
  PC_LAUNCH_CHECK();
  return PC_OK;
}

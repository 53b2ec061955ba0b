// Projected Rayleigh-Ritz problems in FP64 (the FP64 form's iteration and the final step of both
// forms): one CTA per k-point, or a cluster of CTAs where the problems are few (launch_rules.h); the same
// steps as the FP32 kernel (small_rr.cu).
//
// Bound: the FP64 pipe of one SM, two multiply-adds a clock.  A cyclic Jacobi iteration from scratch
// takes some ten sweeps of 6 n^3 FP64 multiply-adds (and as many for V).  So where the basis holds
// search directions (n > m) the matrix C = L^-1 GA L^-H is first diagonalised in FP32 (six sweeps at
// FP32 rates, the replayed rotations give the eigenvectors X of its rounded copy, orthonormal to 1e-6),
// X is made orthonormal in FP64, Q = X (I - E/2 + 3/8 E^2) with E = X^H X - I (orthonormal_factor), and
// C' = Q^H C Q, diagonal to 1e-7, takes one or two FP64 sweeps; Q is orthonormal to FP64's rounding, so the
// result is that of the FP64 iteration (same convergence test, same floor).  A problem whose X is further off
// than that series reaches (overflow or NaN in FP32 among them) is diagonalised from C itself.
// Rayleigh-Ritz of Ritz vectors (n = m) is nearly diagonal already and goes to FP64 directly.
//
// With the conjugate directions, per launch of the reference solves' problems (4 to 6): n = 48 5.6 -> 1.5 ms,
// n = 30 2.4 -> 0.56 ms; n = 72 18 -> 5.6 ms.  What is left: products 0.35, the FP64 sweep 0.33, FP32 stage 0.19,
// factorisations 0.35, conjugate directions 0.17 ms at n = 48.
//
// Two FP64 matrices (72 x 74 complex) and one FP32 matrix fit in shared memory; L, Q and E pass
// through global scratch (L2), as do the logged rotations.
#include <algorithm>
#include <cooperative_groups.h>
#include "jacobi.cuh"
#include "launch_rules.h"

namespace cg = cooperative_groups;

namespace {
constexpr int S6_THREADS = 800;  // 25 warps: 4 for the planes, 21 for the 2 x 2 blocks at n = 72
constexpr int S6_PB = 4;         // panel / row-block width (registers)
constexpr int S6_CLUSTER = kRr64Cluster;  // CTAs per problem where these are few

// Z = A B (herm: A^H B) for n x n matrices, or its upper triangle, in 2 x 2 tiles, up to two per thread
// (n <= 72: 1296 tiles), which fill the lanes whatever n is; store(i, j, z) runs after every product is
// done, so the result may replace an operand.
template <bool UPPER, typename F>
__device__ __forceinline__ void tiles(int n, const double2* A, int lda, bool herm, const double2* B, int ldb, F store) {
  const int h = (n + 1) / 2, nt = UPPER ? h * (h + 1) / 2 : h * h;
  double2 z[2][4];
  int ti[2], tj[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int t = threadIdx.x + q * S6_THREADS;
    ti[q] = -1;
    tj[q] = 0;
    if (t < nt) {
      int I = 0, J;
      if (UPPER) {
        int rem = t;
        while (rem >= h - I) { rem -= h - I; ++I; }
        J = I + rem;
      } else {
        I = t / h;
        J = t - I * h;
      }
      ti[q] = I;
      tj[q] = J;
      const int i0 = 2 * I, i1 = min(2 * I + 1, n - 1), j0 = 2 * J, j1 = min(2 * J + 1, n - 1);
#pragma unroll
      for (int e = 0; e < 4; ++e) z[q][e] = make_double2(0.0, 0.0);
#pragma unroll 2
      for (int p = 0; p < n; ++p) {
        double2 a0 = herm ? A[p * lda + i0] : A[i0 * lda + p], a1 = herm ? A[p * lda + i1] : A[i1 * lda + p];
        if (herm) { a0.y = -a0.y; a1.y = -a1.y; }
        const double2 b0 = B[p * ldb + j0], b1 = B[p * ldb + j1];
        cfma(z[q][0], a0, b0);
        cfma(z[q][1], a0, b1);
        cfma(z[q][2], a1, b0);
        cfma(z[q][3], a1, b1);
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 2; ++q)
    if (ti[q] >= 0)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int i = 2 * ti[q] + (e >> 1), j = 2 * tj[q] + (e & 1);
        if (i < n && j < n && (!UPPER || i <= j)) store(i, j, z[q][e]);
      }
  __syncthreads();
}

// One CTA's share of Z = A B (herm: A^H B) or its upper triangle among CL, one output a thread, so that few
// outputs still spread over the four FP64 units of every SM; `between` runs after the last read of an operand.
template <int CL, bool UPPER, typename S, typename F>
__device__ __forceinline__ void share(int rank, int n, const double2* A, int lda, bool herm, const double2* B, int ldb,
                                      S between, F store) {
  const int nt = UPPER ? n * (n + 1) / 2 : n * n, per = (nt + CL - 1) / CL;
  constexpr int Q = (72 * 72 + CL * S6_THREADS - 1) / (CL * S6_THREADS);
  const int hi = min(nt, (rank + 1) * per);
  double2 z[Q];
  int ti[Q], tj[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    int t = rank * per + threadIdx.x + q * S6_THREADS;
    z[q] = make_double2(0.0, 0.0);
    ti[q] = -1;
    tj[q] = 0;
    if (t < hi) {
      int i = 0, j;
      if (UPPER) {
        while (t >= n - i) { t -= n - i; ++i; }
        j = i + t;
      } else {
        i = t / n;
        j = t - i * n;
      }
      ti[q] = i;
      tj[q] = j;
#pragma unroll 4
      for (int p = 0; p < n; ++p) {
        double2 a = herm ? A[p * lda + i] : A[i * lda + p];
        if (herm) a.y = -a.y;
        cfma(z[q], a, B[p * ldb + j]);
      }
    }
  }
  between();
#pragma unroll
  for (int q = 0; q < Q; ++q)
    if (ti[q] >= 0) store(ti[q], tj[q], z[q]);
}

}  // namespace

// CL > 1: a cluster of CL CTAs per problem.  CTA 0 does everything but the four n x n products of the FP64
// stage, which it shares with the others: they wait for its next product, copy what has changed of the
// operands from its shared memory, and store their part of the result there.  For problems too few to fill
// the chip (one per k-point): a product is bound by the FP64 unit of the SMs it runs on.
template <int CL>
__global__ __launch_bounds__(S6_THREADS, 1) void k_small_rr64(MatRef<double> GA, MatRef<double> GO, int n, int m,
                                                          double drop_tol, const int* __restrict__ klist,
                                                            double* __restrict__ lam_out, double2* __restrict__ coef,
                                                            double2* __restrict__ cpo, double pdir_abs, int* status,
                                                            unsigned char* scratch, long long stride) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int W = S6_THREADS / 32;
  double2* B0 = (double2*)smem;              // GO -> L -> C (positions) -> T -> C' -> Jacobi buffer 1
  double2* B1 = B0 + SR_MAT;                 // GA -> C -> FP32 Jacobi buffers -> X, Q -> Jacobi buffer 0
  float2* F = (float2*)(B1 + SR_MAT);        // X in FP32 -> E in FP32 -> Y
  Plane<double>* pl = (Plane<double>*)(F + SR_MAT);  // 2 x 36 planes
  double* D = (double*)(pl + 72);            // SR_NMAX
  double* ev = D + SR_NMAX;                  // SR_NMAX: reciprocal diagonal of L, then eigenvalues
  int* drop = (int*)(ev + SR_NMAX);          // SR_NMAX
  int* idx = drop + SR_NMAX;                 // SR_NMAX: position -> coordinate (-1: padding)
  int* perm = idx + SR_NMAX;                 // SR_NMAX
  int* low = perm + SR_NMAX;                 // SR_NMAX
  int* misc = low + SR_NMAX;                 // 8: [0] kept, [4..5] largest entry, [6] product
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int k = blockIdx.x / CL;                   // problem
  const int kp = klist ? klist[k] : k;             // its k-point
  double2* Lg = (double2*)(scratch + k * stride);  // n x n: L
  double2* Qg = Lg + n * n;                        // n x n: Q
  double2* Eg = Qg + n * n;                        // n x n: E, then I - E/2 + 3/8 E^2
  void* logk = Eg + n * n;                         // rotations
  double2* ck = coef + (long long)k * n * m;
  double2* cpk = cpo ? cpo + (long long)k * n * m : nullptr;
  enum { DONE, GRAM_X, X_M, C_Q, QH_T };
  // one of the products, by all CTAs of the cluster: f0, b0, b1: CTA 0's F, B0, B1
  auto product = [&](int what, int rank, int nn, float2* f0, double2* b0, double2* b1, auto between) {
    if (what == GRAM_X)  // E = X^H X - I (upper triangle, mirrored)
      share<CL, true>(rank, nn, B1, SR_LD, true, B1, SR_LD, between, [&](int i, int j, double2 g) {
        if (j == i) g = make_double2(g.x - 1.0, 0.0);
        Eg[i * n + j] = g;
        Eg[j * n + i] = cconj(g);
        f0[i * SR_LD + j] = make_float2((float)g.x, (float)g.y);
        f0[j * SR_LD + i] = make_float2((float)g.x, (float)-g.y);
      });
    else if (what == X_M)  // Q = X M
      share<CL, false>(rank, nn, B1, SR_LD, false, Eg, n, between, [&](int i, int j, double2 v) {
        b1[i * SR_LD + j] = v;
        Qg[i * n + j] = v;
      });
    else if (what == C_Q)  // T = C Q
      share<CL, false>(rank, nn, B0, SR_LD, false, B1, SR_LD, between, [&](int i, int j, double2 v) { b0[i * SR_LD + j] = v; });
    else  // C' = Q^H T (upper triangle)
      share<CL, true>(rank, nn, B1, SR_LD, true, B0, SR_LD, between, [&](int i, int j, double2 v) { b0[i * SR_LD + j] = v; });
  };
  if constexpr (CL > 1) {
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    if (rank > 0) {
      float2* f0 = cl.map_shared_rank(F, 0);
      double2 *b0 = cl.map_shared_rank(B0, 0), *b1 = cl.map_shared_rank(B1, 0);
      int* m0 = cl.map_shared_rank(misc, 0);
      for (;;) {
        cl.sync();  // the next product is announced and its operands stand
        const int what = m0[6], nn = m0[0];
        if (what == DONE) break;
        for (int i = warp; i < nn; i += W)
          for (int j = lane; j < nn; j += 32) {
            const int e = i * SR_LD + j;
            if (what == GRAM_X || what == C_Q) B1[e] = b1[e];
            if (what == C_Q || what == QH_T) B0[e] = b0[e];
          }
        __syncthreads();
        product(what, rank, nn, f0, b0, b1, [&] { cl.sync(); });
        cl.sync();  // the result stands
      }
      cl.sync();  // CTA 0's shared memory has been read
      return;
    }
  }
  auto run = [&](int what) {  // CTA 0: the product by the whole cluster (misc[0] columns)
    if constexpr (CL > 1) {
      cg::cluster_group cl = cg::this_cluster();
      if (tid == 0) misc[6] = what;
      cl.sync();
      if (what == DONE) return;
      product(what, 0, misc[0], F, B0, B1, [&] { cl.sync(); });
      cl.sync();
    }
  };
  // scaling, symmetrised copies
  for (int i = warp; i < n; i += W)
    for (int c = lane; c < n; c += 32) {
      B1[i * SR_LD + c] = GA.at(k, i * n + c);
      B0[i * SR_LD + c] = GO.at(k, i * n + c);
    }
  __syncthreads();
  for (int i = tid; i < n; i += S6_THREADS) {
    const double d = B0[i * SR_LD + i].x;
    D[i] = (d > 0.0 && d == d) ? 1.0 / sqrt(d) : 0.0;
    drop[i] = 0;
  }
  __syncthreads();
  for (int i = warp; i < n; i += W)
    for (int c = i + lane; c < n; c += 32) {  // this thread alone reads and writes (i, c) and (c, i)
      const double2 a1 = B1[i * SR_LD + c], a2 = B1[c * SR_LD + i];
      const double2 b1 = B0[i * SR_LD + c], b2 = B0[c * SR_LD + i];
      const double s = D[i] * D[c] * 0.5;
      const double2 a = make_double2((a1.x + a2.x) * s, (a1.y - a2.y) * s), b = make_double2((b1.x + b2.x) * s, (b1.y - b2.y) * s);
      B1[i * SR_LD + c] = a;
      B0[i * SR_LD + c] = b;
      if (c > i) {
        B1[c * SR_LD + i] = cconj(a);
        B0[c * SR_LD + i] = cconj(b);
      }
    }
  __syncthreads();
  // L, T = L^-1 GA, C = L^-1 T^H (upper triangle), all in place
  block_cholesky<double, S6_PB, S6_THREADS>(B0, n, drop_tol, drop, ev);
  block_forward<double, S6_PB, S6_THREADS>(B0, ev, B1, (double2*)nullptr, n, n, n, 0);
  for (int i = warp; i < n; i += W)
    for (int j = i + lane; j < n; j += 32) {
      const double2 u = B1[i * SR_LD + j], l = B1[j * SR_LD + i];
      B1[i * SR_LD + j] = cconj(l);
      B1[j * SR_LD + i] = cconj(u);
    }
  __syncthreads();
  block_forward<double, S6_PB, S6_THREADS>(B0, ev, B1, (double2*)nullptr, n, n, n, 2);
  if (tid == 0) {
    int kept = 0;
    for (int i = 0; i < n; ++i)
      if (!drop[i]) idx[kept++] = i;
    misc[0] = kept;
    if (kept & 1) idx[kept] = -1;  // padding position
  }
  for (int i = warp; i < n; i += W)  // L, for the coefficients at the end
    for (int c = lane; c <= i; c += 32) Lg[i * n + c] = B0[i * SR_LD + c];
  __syncthreads();
  const int nk_ = misc[0];
  double2* Y = (double2*)F;
  double2* Wc = B0;  // coefficients before scaling, n x m
  if (nk_ < m) {
    // too few independent directions: keep the current block (identity on its first m coordinates)
    for (int t = tid; t < n * m; t += S6_THREADS) {
      const int i = t / m, j = t % m;
      const double2 v = make_double2(i == j ? 1.0 : 0.0, 0.0);
      ck[t] = v;
      B1[t] = v;
    }
    for (int j = tid; j < m; j += S6_THREADS) lam_out[(long long)kp * m + j] = GA.at(k, j * n + j).x / GO.at(k, j * n + j).x;
    if (tid == 0) set_status(status, PC_ENOCONV);
    run(DONE);
  } else {
    const int npad = nk_ + (nk_ & 1), np = npad / 2;
    // the kept coordinates of C, in position order, both triangles
    for (int i = warp; i < npad; i += W)
      for (int j = i + lane; j < npad; j += 32) {
        const int a = idx[i], b = idx[j];
        double2 v = (a < 0 || b < 0) ? make_double2(0.0, 0.0) : B1[a * SR_LD + b];
        if (i == j) v.y = 0.0;
        B0[i * SR_LD + j] = v;
        B0[j * SR_LD + i] = cconj(v);
      }
    // rounding floor: eps * max |a_ii| over the kept coordinates of the current Ritz block
    if (warp == 0) {
      double mx = 0.0;
      for (int p = lane; p < nk_; p += 32)
        if (idx[p] < m) mx = fmax(mx, fabs(B1[idx[p] * SR_LD + idx[p]].x));
      for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      if (lane == 0) *reinterpret_cast<double*>(misc + 4) = mx;
    }
    __syncthreads();
    const double amax = *reinterpret_cast<double*>(misc + 4);
    bool use_q = n > m;
    if (use_q) {
      float2 *Fa = (float2*)B1, *Fb = Fa + SR_MAT;
      for (int i = warp; i < npad; i += W)
        for (int j = i + lane; j < npad; j += 32) {
          const double2 v = B0[i * SR_LD + j];
          Fa[spos(i, j)] = make_float2((float)v.x, (float)v.y);
        }
      __syncthreads();
      const int sw = jacobi_sweeps<float, S6_THREADS>(Fa, Fb, (Plane<float>*)pl, (Plane<float>*)logk, nk_, m,
                                                      (float)(1.1920929e-07 * amax), false, (float*)ev, perm, low, misc);
      const int K = sw * (npad - 1);
      Plane<float>*c0 = (Plane<float>*)Fa, *c1 = (Plane<float>*)Fb;
      if (np <= 16) replay<float, 16, 1, S6_THREADS>((Plane<float>*)logk, K, np, nk_, nk_, perm, c0, c1, F, SR_LD);
      else if (np <= 32) replay<float, 16, 2, S6_THREADS>((Plane<float>*)logk, K, np, nk_, nk_, perm, c0, c1, F, SR_LD);
      else replay<float, 16, 3, S6_THREADS>((Plane<float>*)logk, K, np, nk_, nk_, perm, c0, c1, F, SR_LD);
      for (int i = warp; i < nk_; i += W)
        for (int j = lane; j < nk_; j += 32) {
          const float2 v = F[i * SR_LD + j];
          B1[i * SR_LD + j] = make_double2(v.x, v.y);
        }
      __syncthreads();
      // E = X^H X - I
      if constexpr (CL > 1) {
        run(GRAM_X);
      } else {
        tiles<true>(nk_, B1, SR_LD, true, B1, SR_LD, [&](int i, int j, double2 g) {
          if (j == i) g = make_double2(g.x - 1.0, 0.0);
          Eg[i * n + j] = g;
          Eg[j * n + i] = cconj(g);
          F[i * SR_LD + j] = make_float2((float)g.x, (float)g.y);
          F[j * SR_LD + i] = make_float2((float)g.x, (float)-g.y);
        });
      }
      use_q = orthonormal_factor<S6_THREADS>(F, Eg, n, nk_);
      if (use_q) {
        // Q = X M (in place), T = C Q (in place), C' = Q^H T (upper triangle, in place)
        if constexpr (CL > 1) {
          run(X_M);
          run(C_Q);
          run(QH_T);
        } else {
          tiles<false>(nk_, B1, SR_LD, false, Eg, n, [&](int i, int j, double2 v) {
            B1[i * SR_LD + j] = v;
            Qg[i * n + j] = v;
          });
          tiles<false>(nk_, B0, SR_LD, false, B1, SR_LD, [&](int i, int j, double2 v) { B0[i * SR_LD + j] = v; });
          tiles<true>(nk_, B1, SR_LD, true, B0, SR_LD, [&](int i, int j, double2 v) { B0[i * SR_LD + j] = v; });
        }
      }
    }
    run(DONE);
    // FP64 sweeps
    for (int i = warp; i < npad; i += W)
      for (int j = i + lane; j < npad; j += 32) {
        double2 v = (i < nk_ && j < nk_) ? B0[i * SR_LD + j] : make_double2(0.0, 0.0);
        if (i == j) v.y = 0.0;
        B1[spos(i, j)] = v;
      }
    __syncthreads();
    const int sw = jacobi_sweeps<double, S6_THREADS>(B1, B0, pl, (Plane<double>*)logk, nk_, m,
                                                     2.220446049250313e-16 * amax, true, ev, perm, low, misc);
    for (int j = tid; j < m; j += S6_THREADS) lam_out[(long long)kp * m + j] = ev[perm[j]];
    const int K = sw * (npad - 1);
    Plane<double>*c0 = (Plane<double>*)B1, *c1 = (Plane<double>*)B0;
    const double2* Sf = (K & 1) ? B0 : B1;
    if (np <= 16) replay<double, 16, 1, S6_THREADS>((Plane<double>*)logk, K, np, nk_, m, perm, c0, c1, Y, m, Sf, ev);
    else if (np <= 32) replay<double, 32, 1, S6_THREADS>((Plane<double>*)logk, K, np, nk_, m, perm, c0, c1, Y, m, Sf, ev);
    else replay<double, 32, 2, S6_THREADS>((Plane<double>*)logk, K, np, nk_, m, perm, c0, c1, Y, m, Sf, ev);
    // coefficients D L^-H Q Y on the kept coordinates
    for (int t = tid; t < n * m; t += S6_THREADS) Wc[t] = make_double2(0.0, 0.0);
    for (int i = warp; i < n; i += W)
      for (int c = lane; c <= i; c += 32) B1[i * SR_LD + c] = Lg[i * n + c];
    __syncthreads();
    for (int t = tid; t < nk_ * m; t += S6_THREADS) {
      const int p = t / m, j = t - p * m;
      double2 s = Y[t];
      if (use_q) {
        s = make_double2(0.0, 0.0);
        for (int q = 0; q < nk_; ++q) cfma(s, Qg[p * n + q], Y[q * m + j]);
      }
      Wc[idx[p] * m + j] = s;
    }
    __syncthreads();
    block_backward<double, S6_PB, S6_THREADS>(B1, Wc, m, n, m);
    for (int t = tid; t < n * m; t += S6_THREADS) {
      const double2 c = cscale(Wc[t], D[t / m]);
      ck[t] = c;
      B1[t] = c;  // cX for the conjugate directions
    }
  }
  if (cpk) {
    __syncthreads();
    pdir<double, S6_THREADS>(GO, k, n, m, pdir_abs, B0, B1, B1 + n * m, B1 + 2 * n * m, (double2*)F, (double2*)F + m * (m | 1),
                             ev, drop, cpk);
  }
  if constexpr (CL > 1) cg::this_cluster().sync();  // the others have read this CTA's shared memory
}

// L, Q and E, and the planes (32 bytes) of the rotations of the most sweeps and of the round after them.
long long small_rr64_scratch(int n) {
  return 16LL * 3 * n * n + 32LL * ((long long)SR_MAX_SWEEPS * n + 1) * ((n + 1) / 2);
}

int launch_small_rr64(const MatRef<double>& GA, const MatRef<double>& GO, int n, int m, int nk, double drop_tol, const int* klist,
                      double* lam_out, double2* coef, double2* cp, double pdir_abs, int* status, void* scratch,
                      long long stride, int slots, long long others, cudaStream_t s) {
  if (n > SR_NMAX || m > n || m > 24 || n < 1 || slots < 1 || stride < small_rr64_scratch(n) || stride % 16) return PC_EINVAL;
  const size_t sm = sizeof(double2) * 2 * (size_t)SR_MAT + sizeof(float2) * SR_MAT + sizeof(Plane<double>) * 72 +
                    sizeof(double) * 2 * SR_NMAX + sizeof(int) * (4 * SR_NMAX + 8);
  static const bool clusters =  // once, thread-safe (k groups launch from several host threads)
      cudaFuncSetAttribute(k_small_rr64<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) == cudaSuccess &&
      cudaFuncSetAttribute(k_small_rr64<S6_CLUSTER>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) == cudaSuccess;
  // (4 problems, n = 48, as the iteration calls it: 1.17 ms by one CTA each, 1.0 by clusters; the same bits)
  const bool cluster = clusters && rr64_uses_clusters(n, m, nk, others, device_sms());
  for (int f = 0; f < nk; f += slots) {
    const int count = std::min(slots, nk - f);
    const MatRef<double> ga = GA.from(f), go = GO.from(f);
    const int* kl = klist ? klist + f : nullptr;
    double* lam = klist ? lam_out : lam_out + (long long)f * m;
    const long long o = (long long)f * n * m;
    double2 *cx = coef + o, *cpf = cp ? cp + o : nullptr;
    bool launched = false;
    if (cluster) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(count * S6_CLUSTER);
      cfg.blockDim = dim3(S6_THREADS);
      cfg.dynamicSmemBytes = sm;
      cfg.stream = s;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = S6_CLUSTER;
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      launched = cudaLaunchKernelEx(&cfg, k_small_rr64<S6_CLUSTER>, ga, go, n, m, drop_tol, kl, lam, cx, cpf, pdir_abs,
                                    status, (unsigned char*)scratch, stride) == cudaSuccess;
      if (!launched) cudaGetLastError();  // no room for a cluster here: one CTA per problem
    }
    if (!launched)
      k_small_rr64<1><<<count, S6_THREADS, sm, s>>>(ga, go, n, m, drop_tol, kl, lam, cx, cpf, pdir_abs, status,
                                                    (unsigned char*)scratch, stride);
    PC_LAUNCH_CHECK();
  }
  return PC_OK;
}

// The condensed operator A(k) = H Phi^-1 H^* of eq. matrixform, applied to blocks of
// vectors at every k, and the block iteration's residual / preconditioner kernels.
//
// With H block diagonal in the plane-wave index (the centroid sum of a non-zero
// plane-wave difference vanishes when n_i >= 2M+1) and an isotropic compliance, the
// stress space splits into one bulk and five deviatoric orthonormal tensor
// coordinates.  The compliance acts as f1 on the bulk coordinate and f2 on the five
// deviatoric ones, so
//     A(k) U = (2 pi V)^2 sum_s B_s(K)^T W_s B_s(K) U,   W_0 = T_f1^-1, W_1..5 = T_f2^-1,
// where B_s(K_q) maps the displacement coefficients at wave q to coordinate s of the
// symmetric gradient sym(K_q (x) u).  Applying A is three steps: form the six strain
// stacks (B), multiply by the k-independent W (one GEMM over all k and vectors), and
// contract back with B (epilogue).
#include "kernels.h"
#include "waves.cuh"

// Wavevectors of a set of k-points in FP32, Kf[k N + q] = (K_0, K_1, K_2, 0) of plane wave q:
// computed in FP64 by kvec and rounded, as the FP32 kernels would round them; they read the
// table instead of recomputing (FP64 arithmetic and two integer divisions per element).
__global__ void k_kvec_table(Geom g, const double* __restrict__ Q, int nk, float4* __restrict__ Kf) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)nk * g.N) return;
  const int k = (int)(t / g.N), q = (int)(t % g.N);
  double K[3];
  kvec(g, Q, k, q, K);
  Kf[t] = make_float4((float)K[0], (float)K[1], (float)K[2], 0.f);
}
int launch_kvec_table(Geom g, const double* Q, int nk, float4* Kf, cudaStream_t s) {
  const long long n = (long long)nk * g.N;
  if (n == 0) return PC_OK;
  k_kvec_table<<<cdiv(n, 256), 256, 0, s>>>(g, Q, nk, Kf);
  PC_LAUNCH_CHECK();
  return PC_OK;
}

// ---------------------------------------------------------------------------
// Complex GEMMs on CUDA cores, up to three products of the same row count and depth in one launch:
// C[col][p] = alpha * sum_q A[p][q] * B[col][q].  16 U x 16 U output tile, 16-deep K slices staged in
// shared memory, U x U outputs per thread, each accumulated over q in order.
//
// Bound (FP64): the two multiply-adds a clock of an SM's FP64 pipe; staging costs nothing beside it at
// any U.  So the tile is the one whose busiest SM has the least work, ceil(tiles / SMs) x tile area: the
// operator of a reference solve (N = 125, 64 vectors) is 18 tiles of 64 x 64 in three launches on 152 SMs
// (1.55 ms an application) but 288 of 16 x 16 in one (0.067 ms); N = 343 with 48 vectors 4.2 -> 0.36 ms.
template <typename R> struct GemmSegs {
  GemmSeg<R> s[3];
  int tile0[4];  // first column tile of each product, and their total
};
template <typename R, int U>
__global__ __launch_bounds__(256) void k_gemm(int Mrows, int K, int lda, long long ldb, long long ldc, GemmSegs<R> segs) {
  typedef typename cplx_t<R>::type C2;
  constexpr int T = 16 * U;
  __shared__ C2 As[16][T + 1];
  __shared__ C2 Bs[16][T + 1];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int g = ((int)blockIdx.x >= segs.tile0[1]) + ((int)blockIdx.x >= segs.tile0[2]);
  const GemmSeg<R> sg = segs.s[g];
  const int p0 = blockIdx.y * T;
  const long long c0 = (long long)((int)blockIdx.x - segs.tile0[g]) * T;
  C2 acc[U][U];
  const C2* bcol[U];  // this thread's columns of B (row r = threadIdx.x / 16 + 16 i of the tile)
#pragma unroll
  for (int i = 0; i < U; ++i) {
    const long long col = c0 + (threadIdx.x >> 4) + 16 * i;
    bcol[i] = col < sg.ncols ? sg.B + sg.column(col) * ldb : nullptr;
#pragma unroll
    for (int j = 0; j < U; ++j) acc[i][j] = mk<R>(0, 0);
  }
  for (int k0 = 0; k0 < K; k0 += 16) {
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const int r = (threadIdx.x >> 4) + 16 * i, kk = threadIdx.x & 15;
      const int p = p0 + r, q = k0 + kk;
      As[kk][r] = (p < Mrows && q < K) ? sg.A[(long long)p * lda + q] : mk<R>(0, 0);
      Bs[kk][r] = (bcol[i] && q < K) ? bcol[i][q] : mk<R>(0, 0);
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      C2 a[U], b[U];
#pragma unroll
      for (int i = 0; i < U; ++i) a[i] = As[kk][tx + 16 * i];
#pragma unroll
      for (int j = 0; j < U; ++j) b[j] = Bs[kk][ty + 16 * j];
#pragma unroll
      for (int i = 0; i < U; ++i)
#pragma unroll
        for (int j = 0; j < U; ++j) cfma(acc[i][j], a[i], b[j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < U; ++j) {
    long long col = c0 + ty + 16 * j;
    if (col >= sg.ncols) continue;
    const long long out = sg.column(col) * ldc;
#pragma unroll
    for (int i = 0; i < U; ++i) {
      int p = p0 + tx + 16 * i;
      if (p < Mrows) sg.C[out + p] = cscale(acc[i][j], sg.alpha);
    }
  }
}

int device_sms() {
  static const int n = [] {  // queried once; thread-safe static initialisation
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 152;
    cudaGetLastError();
    return v;
  }();
  return n;
}

template <typename R>
int launch_gemms(int Mrows, int K, int lda, long long ldb, long long ldc, const GemmSeg<R>* seg, int nseg, cudaStream_t s) {
  if (nseg < 1 || nseg > 3 || Mrows < 1) return PC_EINVAL;
  int best = 4;
  long long best_t = -1;
  for (int u = 4; u >= 1; u >>= 1) {
    const long long T = 16 * u;
    long long tiles = 0;
    for (int g = 0; g < nseg; ++g) tiles += (seg[g].ncols + T - 1) / T;
    tiles *= cdiv(Mrows, T);
    const long long t = (tiles + device_sms() - 1) / device_sms() * T * T;
    if (best_t < 0 || t < best_t) { best_t = t; best = u; }
  }
  GemmSegs<R> a;
  int tiles = 0;
  for (int g = 0; g < 3; ++g) {
    a.s[g] = seg[g < nseg ? g : nseg - 1];
    a.tile0[g] = tiles;
    if (g < nseg) tiles += cdiv(seg[g].ncols, 16 * best);
    else a.tile0[g] = 0x7fffffff;
  }
  a.tile0[3] = tiles;
  if (tiles == 0) return PC_OK;
  const dim3 grid(tiles, cdiv(Mrows, 16 * best));
  if (best == 4) k_gemm<R, 4><<<grid, 256, 0, s>>>(Mrows, K, lda, ldb, ldc, a);
  else if (best == 2) k_gemm<R, 2><<<grid, 256, 0, s>>>(Mrows, K, lda, ldb, ldc, a);
  else k_gemm<R, 1><<<grid, 256, 0, s>>>(Mrows, K, lda, ldb, ldc, a);
  PC_LAUNCH_CHECK();
  return PC_OK;
}
template int launch_gemms<double>(int, int, int, long long, long long, const GemmSeg<double>*, int, cudaStream_t);
template int launch_gemms<float>(int, int, int, long long, long long, const GemmSeg<float>*, int, cudaStream_t);

// ---------------------------------------------------------------------------
// Strain stacks: E[s][vec][q] = sum_c B_s(K_q)[c] U[vec][c][q].
template <typename R>
__global__ void k_strain(const typename cplx_t<R>::type* __restrict__ X, int nvec, int m, Geom g,
                         const double* __restrict__ Q, const float4* __restrict__ Kf,
                         typename cplx_t<R>::type* __restrict__ E, VecSel sel) {
  typedef typename cplx_t<R>::type C2;
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int N = g.N;
  if (t >= (long long)nvec * N) return;
  const int vec = sel((int)(t / N)), q = (int)(t % N);
  R k0, k1, k2;
  kvec_r<R>(g, Q, Kf, vec / m, q, k0, k1, k2);
  const C2* x = X + (long long)vec * 3 * N;
  const long long st = (long long)nvec * N;
  C2 e[6];
  strain6<R>(k0, k1, k2, x[q], x[N + q], x[2 * N + q], e);
#pragma unroll
  for (int i = 0; i < 6; ++i) E[i * st + t] = e[i];
}
template <typename R>
int launch_strain(const typename cplx_t<R>::type* X, int nvec, int m, Geom g, const double* Q,
                  typename cplx_t<R>::type* E, cudaStream_t s, const float4* Kf, VecSel sel) {
  long long n = (long long)nvec * g.N;
  if (sizeof(R) != sizeof(float)) Kf = nullptr;  // the table is FP32
  if (n == 0) return PC_OK;
  k_strain<R><<<cdiv(n, 256), 256, 0, s>>>(X, nvec, m, g, Q, Kf, E, sel);
  PC_LAUNCH_CHECK();
  return PC_OK;
}
template int launch_strain<double>(const double2*, int, int, Geom, const double*, double2*, cudaStream_t, const float4*, VecSel);
template int launch_strain<float>(const float2*, int, int, Geom, const double*, float2*, cudaStream_t, const float4*, VecSel);

// Epilogue: AX[vec][c][p] = sum_s c_s B_s(K_p)[c] Sig[s][vec][p]   (c_0 bulk, c_1 deviatoric).
template <typename R>
__global__ void k_epilogue(const typename cplx_t<R>::type* __restrict__ S, int nvec, int m, Geom g,
                           const double* __restrict__ Q, const float4* __restrict__ Kf, R c0, R c1,
                           typename cplx_t<R>::type* __restrict__ AX, VecSel sel) {
  typedef typename cplx_t<R>::type C2;
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int N = g.N;
  if (t >= (long long)nvec * N) return;
  const int vec = sel((int)(t / N)), p = (int)(t % N);
  R k0, k1, k2;
  kvec_r<R>(g, Q, Kf, vec / m, p, k0, k1, k2);
  const long long st = (long long)nvec * N;
  C2 o[3];
  strain6_t<R>(k0, k1, k2, S + t, st, c0, c1, o);
  C2* out = AX + (long long)vec * 3 * N + p;
  out[0] = o[0]; out[N] = o[1]; out[2 * N] = o[2];
}
template <typename R>
int launch_epilogue(const typename cplx_t<R>::type* Sig, int nvec, int m, Geom g, const double* Q,
                    R c0, R c1, typename cplx_t<R>::type* AX, cudaStream_t s, const float4* Kf, VecSel sel) {
  long long n = (long long)nvec * g.N;
  if (sizeof(R) != sizeof(float)) Kf = nullptr;  // the table is FP32
  if (n == 0) return PC_OK;
  k_epilogue<R><<<cdiv(n, 256), 256, 0, s>>>(Sig, nvec, m, g, Q, Kf, c0, c1, AX, sel);
  PC_LAUNCH_CHECK();
  return PC_OK;
}
template int launch_epilogue<double>(const double2*, int, int, Geom, const double*, double, double, double2*, cudaStream_t, const float4*, VecSel);
template int launch_epilogue<float>(const float2*, int, int, Geom, const double*, float, float, float2*, cudaStream_t, const float4*, VecSel);

// ---------------------------------------------------------------------------
// Relative residuals ||A x - lambda Omega x|| / (max(|lambda|, floor) ||Omega x||), one block per vector.
// The floor is 1e-2 of the largest wanted eigenvalue at that k (zero modes at Gamma).
template <typename R>
__global__ void k_resnorm(const typename cplx_t<R>::type* __restrict__ AX, const typename cplx_t<R>::type* __restrict__ OX,
                          const R* __restrict__ lam, int m, int nb, int n3, double tol, double* __restrict__ rnorm,
                          int* __restrict__ active, const int* __restrict__ klist) {
  typedef typename cplx_t<R>::type C2;
  __shared__ double ra[256], rb[256];
  const int k = klist ? klist[blockIdx.x / m] : (int)blockIdx.x / m;
  const int vec = k * m + (int)blockIdx.x % m;
  R l = lam[vec];
  const C2* ax = AX + (long long)vec * n3;
  const C2* ox = OX + (long long)vec * n3;
  R sa = 0, sb = 0;  // per-thread partial sums in the block's own precision
  for (int r = threadIdx.x; r < n3; r += blockDim.x) {
    C2 a = ax[r], o = ox[r];
    R dx = a.x - l * o.x, dy = a.y - l * o.y;
    sa += dx * dx + dy * dy;
    sb += o.x * o.x + o.y * o.y;
  }
  ra[threadIdx.x] = (double)sa;
  rb[threadIdx.x] = (double)sb;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) { ra[threadIdx.x] += ra[threadIdx.x + w]; rb[threadIdx.x] += rb[threadIdx.x + w]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    double lmax = fabs((double)lam[k * m + nb - 1]);
    double scale = fmax(fabs((double)l), 1e-2 * lmax);
    double rn = (rb[0] > 0.0 && scale > 0.0) ? sqrt(ra[0]) / (scale * sqrt(rb[0])) : 0.0;
    if (!(rn == rn)) rn = 1e300;
    rnorm[vec] = rn;
    active[vec] = rn > tol ? 1 : 0;
  }
}
// The convergence test of the open k-points (in klist order, `nopen` of them, or all nk without a list),
// by one CTA.  A k-point whose wanted bands are all below tolerance is locked for good (kdone = 1): its
// block is no longer updated.
// The target is 0.4 of the tolerance, and a k-point below the tolerance gets one more iteration to reach it: the
// preconditioner takes the short waves out of a residual, so that one at the tolerance says less about the
// vectors than one that a plane-wave resolvent leaves.  Gradients of randomly weighted bands of the 8^3 cube
// cells, tolerance 3e-4: errors of 2.9e-5 to 16e-5 with the resolvent alone, 3.3e-5 to 11e-5 with the products
// and no margin, 2.7e-5 to 5.7e-5 at half the tolerance, for none to one iteration in fourteen.  Design steps at
// 1e-4: half the resolvent's errors (0.4 to 2.3e-6 instead of 1.2 to 3e-6); 0.4 is 12 % below half, for 1 % of the time.
// Stagnation: the carried FP32 products A X and Omega X drift by rounding, so a k-point's
// residual can settle at an attainable floor a little above the tolerance.  A k-point whose
// worst wanted residual has not dropped below 0.95 of its best for STALL_ITERS iterations and
// lies within STALL_FACTOR times the tolerance is accepted at that floor.
// The lists of the next iteration come out compacted and in order; klist is read before it is rewritten
// (a chunk's outputs never pass the inputs already read).
#define STALL_ITERS 20
#define STALL_FACTOR 10.0
#define TARGET 0.4
__global__ __launch_bounds__(256) void k_open(const int* __restrict__ active, const double* __restrict__ rnorm, double tol,
                                              int nopen, int m, int nb, int* __restrict__ kdone, double* __restrict__ best,
                                              int* __restrict__ since, OpenSet o, int lists) {
  __shared__ int sums[4][8], base[4];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid < 4) base[tid] = 0;
  __syncthreads();
  for (int p0 = 0; p0 < nopen; p0 += 256) {
    const int p = p0 + tid;
    int k = -1, open = 0, fresh = 0, cols = 0, above = 0;
    if (p < nopen) {
      k = lists ? o.klist[p] : p;
      int a = 0;
      double worst = 0.0;
      for (int j = 0; j < m; ++j) {
        const int aj = active[k * m + j];
        cols += aj;
        if (j < nb) {
          a |= aj;
          worst = fmax(worst, rnorm[k * m + j]);
        }
      }
      bool done = !a;
      if (!done && worst <= tol) {
        done = kdone[k] == 2;  // the second time
        kdone[k] = 2;
      } else if (best && !done) {
        if (best[k] == 0.0 || worst < 0.95 * best[k]) {
          best[k] = worst;
          since[k] = 0;
        } else if (++since[k] >= STALL_ITERS && worst <= STALL_FACTOR * tol) {
          done = true;
        }
      }
      if (done || kdone[k] != 2) kdone[k] = done ? 1 : 0;
      open = done ? 0 : 1;
      fresh = done ? 1 : 0;
      above = open && worst > tol ? 1 : 0;
      if (done) cols = 0;
    }
    int v[4] = {open, cols, fresh, above}, x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x[i] = v[i];
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x[i], d);
        if (lane >= d) x[i] += y;
      }
      if (lane == 31) sums[i][warp] = x[i];
    }
    __syncthreads();  // also: every k of this chunk has been read
    int off[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      off[i] = base[i] + x[i] - v[i];
      for (int w = 0; w < warp; ++w) off[i] += sums[i][w];
    }
    if (lists && k >= 0) {
      if (open) o.klist[off[0]] = k;
      if (fresh) o.fresh[off[2]] = k;
      if (open)
        for (int j = 0; j < m; ++j) {
          o.vpos[k * m + j] = active[k * m + j] ? off[1] : -1;
          if (active[k * m + j]) o.vlist[off[1]++] = k * m + j;
        }
    }
    __syncthreads();
    if (tid < 4)
      for (int w = 0; w < 8; ++w) base[tid] += sums[tid][w];
    __syncthreads();
  }
  if (tid < 4) o.count[tid] = base[tid];
}
// All k-points open; and the reference medium of the preconditioner, from the mean chi.
__global__ void k_open_all(int* klist, int nk, PrecRef pr, const double* __restrict__ chi_mean, double* __restrict__ ref) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < nk) klist[k] = k;
  if (k != 0) return;
  const double cm = *chi_mean;
  // 3 kappa and 2 mu: of the material with the mean compliance, with the mean Lame constants, or the
  // geometric mean of the two (softest, stiffest and between)
  const double s1 = 1.0 / (pr.f1_0 + cm * (pr.f1_1 - pr.f1_0)), s2 = 1.0 / (pr.f2_0 + cm * (pr.f2_1 - pr.f2_0));
  const double mu = pr.mu0 + cm * (pr.mu1 - pr.mu0), la = pr.lam0 + cm * (pr.lam1 - pr.lam0);
  const double t1 = 3.0 * la + 2.0 * mu, t2 = 2.0 * mu;
  const double w1 = pr.ref_mode == 1 ? s1 : (pr.ref_mode == 0 ? t1 : sqrt(s1 * t1));
  const double w2 = pr.ref_mode == 1 ? s2 : (pr.ref_mode == 0 ? t2 : sqrt(s2 * t2));
  ref[0] = pr.two_pi_sq_V_over_sA * w1;
  ref[1] = pr.two_pi_sq_V_over_sA * w2;
  ref[2] = pr.half_lref_V_over_sA * (pr.rho0 + cm * (pr.rho1 - pr.rho0)) * pr.shift_scale;
}
int launch_open_all(OpenSet o, int nk, PrecRef pr, const double* chi_mean, double* ref, cudaStream_t s) {
  k_open_all<<<cdiv(nk, 256), 256, 0, s>>>(o.klist, nk, pr, chi_mean, ref);
  PC_LAUNCH_CHECK();
  return PC_OK;
}
template <typename R>
int launch_resnorm(const typename cplx_t<R>::type* AX, const typename cplx_t<R>::type* OX, const R* lam,
                   int nk, int m, int nb, int n3, double tol, double* rnorm, int* active, int* kdone, OpenSet o, int nopen,
                   cudaStream_t s, double* best, int* since) {
  const int lists = o.klist != nullptr;
  const int n = lists ? nopen : nk;
  k_resnorm<R><<<n * m, 256, 0, s>>>(AX, OX, lam, m, nb, n3, lists ? TARGET * tol : tol, rnorm, active, o.klist);
  PC_LAUNCH_CHECK();
  k_open<<<1, 256, 0, s>>>(active, rnorm, tol, n, m, nb, kdone, best, since, o, lists);
  PC_LAUNCH_CHECK();
  return PC_OK;
}
template int launch_resnorm<double>(const double2*, const double2*, const double*, int, int, int, int, double, double*, int*, int*, OpenSet, int, cudaStream_t, double*, int*);
template int launch_resnorm<float>(const float2*, const float2*, const float*, int, int, int, int, double, double*, int*, int*, OpenSet, int, cudaStream_t, double*, int*);

// First half of the preconditioner (waves.cuh) on the unconverged columns: Y = R0 (A x - lambda Omega x) into
// W, and its strain stacks E[s][v][q], v counting along vlist.
template <typename R>
__global__ void k_prec_in(const typename cplx_t<R>::type* __restrict__ AX, const typename cplx_t<R>::type* __restrict__ OX,
                          const R* __restrict__ lam, const int* __restrict__ vlist, int nvec, int m, int nb, Geom g,
                          const double* __restrict__ Q, const float4* __restrict__ Kf, const double* __restrict__ ref,
                          typename cplx_t<R>::type* __restrict__ W, typename cplx_t<R>::type* __restrict__ E) {
  typedef typename cplx_t<R>::type C2;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int N = g.N;
  if (t >= (long long)nvec * N) return;
  const int vec = vlist[(int)(t / N)], q = (int)(t % N), k = vec / m;
  C2 u[3], e[6];
  prec_residual<R>(PrecTerm<R>(ref, lam + k * m, nb), AX, OX, W, lam[vec], vec, g, Q, Kf, k, q, u, e);
  const long long st = (long long)nvec * N;
#pragma unroll
  for (int i = 0; i < 6; ++i) E[i * st + t] = e[i];
}
// Second half: W = R0 [B^T W0 S + s Y] with S = T W0 B Y (T E, the moduli applied here) on the unconverged
// columns of the open k-points; W = A W = Omega W = 0 on the others (the operator is applied to the former only).
template <typename R>
__global__ void k_prec_out(const typename cplx_t<R>::type* __restrict__ S, const R* __restrict__ lam,
                           const int* __restrict__ klist, const int* __restrict__ vpos, int nall, int nvec, int m, int nb,
                           Geom g, const double* __restrict__ Q, const float4* __restrict__ Kf,
                           const double* __restrict__ ref, typename cplx_t<R>::type* __restrict__ W,
                           typename cplx_t<R>::type* __restrict__ AW, typename cplx_t<R>::type* __restrict__ OW) {
  typedef typename cplx_t<R>::type C2;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int N = g.N;
  if (t >= (long long)nall * N) return;
  const int v = (int)(t / N), q = (int)(t % N), k = klist[v / m], vec = k * m + v % m, pos = vpos[vec];
  const long long o = (long long)vec * 3 * N + q;
  C2* w = W + o;
  if (pos < 0) {
    C2 *aw = AW + o, *ow = OW + o;
    for (int c = 0; c < 3; ++c) w[c * N] = aw[c * N] = ow[c * N] = mk<R>(0, 0);
    return;
  }
  const PrecTerm<R> pt(ref, lam + k * m, nb);
  R k0, k1, k2;
  kvec_r<R>(g, Q, Kf, k, q, k0, k1, k2);
  C2 z[3];
  strain6_t<R>(k0, k1, k2, S + (long long)pos * N + q, (long long)nvec * N, pt.w1 * pt.w1, pt.w2 * pt.w2, z);
#pragma unroll
  for (int c = 0; c < 3; ++c) z[c] = mk<R>(z[c].x + pt.s * w[c * N].x, z[c].y + pt.s * w[c * N].y);
  pt.solve(k0, k1, k2, z);
  for (int c = 0; c < 3; ++c) w[c * N] = z[c];
}
template <typename R>
int launch_prec_in(const typename cplx_t<R>::type* AX, const typename cplx_t<R>::type* OX, const R* lam, const int* vlist,
                   int ncol, int m, int nb, Geom g, const double* Q, const double* ref, typename cplx_t<R>::type* W,
                   typename cplx_t<R>::type* E, cudaStream_t s, const float4* Kf) {
  if (sizeof(R) != sizeof(float)) Kf = nullptr;  // the table is FP32
  k_prec_in<R><<<cdiv((long long)ncol * g.N, 256), 256, 0, s>>>(AX, OX, lam, vlist, ncol, m, nb, g, Q, Kf, ref, W, E);
  PC_LAUNCH_CHECK();
  return PC_OK;
}
template <typename R>
int launch_prec_out(const typename cplx_t<R>::type* S, const R* lam, const int* klist, const int* vpos, int nopen, int ncol,
                    int m, int nb, Geom g, const double* Q, const double* ref, typename cplx_t<R>::type* W,
                    typename cplx_t<R>::type* AW, typename cplx_t<R>::type* OW, cudaStream_t s, const float4* Kf) {
  if (sizeof(R) != sizeof(float)) Kf = nullptr;
  k_prec_out<R><<<cdiv((long long)nopen * m * g.N, 256), 256, 0, s>>>(S, lam, klist, vpos, nopen * m, ncol, m, nb, g, Q, Kf,
                                                                      ref, W, AW, OW);
  PC_LAUNCH_CHECK();
  return PC_OK;
}
template int launch_prec_in<double>(const double2*, const double2*, const double*, const int*, int, int, int, Geom, const double*, const double*, double2*, double2*, cudaStream_t, const float4*);
template int launch_prec_in<float>(const float2*, const float2*, const float*, const int*, int, int, int, Geom, const double*, const double*, float2*, float2*, cudaStream_t, const float4*);
template int launch_prec_out<double>(const double2*, const double*, const int*, const int*, int, int, int, int, Geom, const double*, const double*, double2*, double2*, double2*, cudaStream_t, const float4*);
template int launch_prec_out<float>(const float2*, const float*, const int*, const int*, int, int, int, int, Geom, const double*, const double*, float2*, float2*, float2*, cudaStream_t, const float4*);

template <typename R>
__global__ void k_store(const typename cplx_t<R>::type* __restrict__ src, double2* __restrict__ dst,
                        const int* __restrict__ list, long long per) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < per) dst[list[blockIdx.y] * per + t] = to_d2(src[list[blockIdx.y] * per + t]);
}
template <typename R>
int launch_store(const typename cplx_t<R>::type* src, double2* dst, const int* list, int nsel, long long per, cudaStream_t s) {
  if (nsel <= 0) return PC_OK;
  k_store<R><<<dim3(cdiv(per, 256), nsel), 256, 0, s>>>(src, dst, list, per);
  PC_LAUNCH_CHECK();
  return PC_OK;
}
template int launch_store<double>(const double2*, double2*, const int*, int, long long, cudaStream_t);
template int launch_store<float>(const float2*, double2*, const int*, int, long long, cudaStream_t);

// ---------------------------------------------------------------------------
// Initial block: the m lowest homogeneous plane waves (ranked by |K_q|, ties by index),
// one displacement component each, plus a 1e-3 counter-hash perturbation on every entry
// so that no exact degeneracy of the start block survives.  The perturbation depends on
// (band, component, wave) only, so equal wavevectors get bitwise equal results.
__device__ __forceinline__ double hash_unit(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  x = x ^ (x >> 31);
  return (double)(x >> 11) * (1.0 / 9007199254740992.0) * 2.0 - 1.0;
}
// The |K|^2 of the k-point's waves are computed once per CTA and compared on the integer units (they are not
// negative, so their bits order as they do): with both in FP64 for every pair of waves, N^2 a k-point, N = 729
// took 2.08 ms for 50 k-points (now 0.12).  A wave whose rank is past the block stops counting.
template <typename R>
__global__ __launch_bounds__(256) void k_init_guess(typename cplx_t<R>::type* __restrict__ X, int nk, int m, Geom g,
                                                    const double* __restrict__ Q, unsigned long long seed) {
  extern __shared__ long long ksq[];
  const int k = blockIdx.y;
  const int N = g.N;
  for (int p = threadIdx.x; p < N; p += blockDim.x) {
    double K[3];
    kvec(g, Q, k, p, K);
    ksq[p] = __double_as_longlong(K[0] * K[0] + K[1] * K[1] + K[2] * K[2]);
  }
  __syncthreads();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= N) return;
  const long long kq = ksq[q];
  const int last = (m - 1) / 3;
  int rank = 0;
  for (int p = 0; p < N && rank <= last; ++p) rank += (ksq[p] < kq || (ksq[p] == kq && p < q)) ? 1 : 0;
  for (int j = 0; j < m; ++j) {
    for (int c = 0; c < 3; ++c) {
      long long idx = ((long long)(k * m + j) * 3 + c) * N + q;
      unsigned long long h = (((unsigned long long)j * 3ull + c) * (unsigned long long)N + q) * 2ull + seed * 0x100000000ull;
      double v = 1e-3 * hash_unit(h), w = 1e-3 * hash_unit(h + 1);
      if (j / 3 == rank && j % 3 == c) v += 1.0;
      X[idx] = mk<R>((R)v, (R)w);
    }
  }
}
template <typename R>
int launch_init_guess(typename cplx_t<R>::type* X, int nk, int m, Geom g, const double* Q, unsigned long long seed,
                      cudaStream_t s) {
  dim3 grid(cdiv(g.N, 256), nk);
  k_init_guess<R><<<grid, 256, sizeof(long long) * g.N, s>>>(X, nk, m, g, Q, seed);
  PC_LAUNCH_CHECK();
  return PC_OK;
}
template int launch_init_guess<double>(double2*, int, int, Geom, const double*, unsigned long long, cudaStream_t);
template int launch_init_guess<float>(float2*, int, int, Geom, const double*, unsigned long long, cudaStream_t);

__global__ void k_f2d(const float2* __restrict__ s, double2* __restrict__ d, long long n) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) d[t] = make_double2(s[t].x, s[t].y);
}
int launch_convert_f2d(const float2* src, double2* dst, long long n, cudaStream_t s) {
  k_f2d<<<cdiv(n, 256), 256, 0, s>>>(src, dst, n);
  PC_LAUNCH_CHECK();
  return PC_OK;
}

__global__ void k_d2f(const double2* __restrict__ s, float2* __restrict__ d, long long n, double scale) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) d[t] = make_float2((float)(s[t].x * scale), (float)(s[t].y * scale));
}
int launch_d2f(const double2* src, float2* dst, long long n, double scale, cudaStream_t s) {
  k_d2f<<<cdiv(n, 256), 256, 0, s>>>(src, dst, n, scale);
  PC_LAUNCH_CHECK();
  return PC_OK;
}

__global__ void k_scale_d2(double2* __restrict__ x, long long n, double s) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) { x[t].x *= s; x[t].y *= s; }
}
int launch_scale_d2(double2* x, long long n, double s, cudaStream_t st) {
  k_scale_d2<<<cdiv(n, 256), 256, 0, st>>>(x, n, s);
  PC_LAUNCH_CHECK();
  return PC_OK;
}

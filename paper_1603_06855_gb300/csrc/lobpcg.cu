// Batched block operations of the locally optimal block preconditioned conjugate
// gradient iteration (one independent problem per k-point), and the small projected
// problems solved one CTA per k:
//   gram   -- G = A^H B over the 3N rows, for up to three m-column blocks per side
//   update -- out = [S_0 S_1 S_2] C for up to three operand triplets sharing C
//   small_chol -- Cholesky-QR transform T with T^H G T = I (dependent columns -> zero)
#include <type_traits>
#include "kernels.h"
#include "small_dense.cuh"

#define GRAM_SPLIT 8
#define GRAM_LD 73   // odd row stride of the shared tiles (columns up to 72)


// G_part[k][split] = A^H B over one row range; each of the 16 x 16 threads holds TILE x TILE outputs.  Shared tiles are double-buffered: the next
// tile of GRAM_ROWS rows (16 in FP32, 8 in FP64: 37 KB of static shared memory either way)
// is fetched into registers while the current one is multiplied.
template <typename R, typename RA, int TILE>
__global__ __launch_bounds__(256) void k_gram(BlockList<R> A, int na, BlockList<R> B, int nbk, int m, int n3,
                                              typename cplx_t<R>::type* __restrict__ part) {
  typedef typename cplx_t<R>::type C2;
  typedef typename cplx_t<RA>::type CA;
  constexpr int GRAM_ROWS = sizeof(R) == 8 ? 8 : 16;
  __shared__ C2 sA[2][GRAM_ROWS * GRAM_LD];
  __shared__ C2 sB[2][GRAM_ROWS * GRAM_LD];
  const int k = blockIdx.x, split = blockIdx.y;
  const int ca = na * m, cb = nbk * m;
  const long long kofs = (long long)k * m * n3;
  const int chunk = (n3 + GRAM_SPLIT - 1) / GRAM_SPLIT;
  const int r_begin = split * chunk, r_end = min(n3, r_begin + chunk);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  // each thread stages elements t = threadIdx.x + 256 u of the (rows x cols) tiles
  const int nla = (GRAM_ROWS * ca + 255) / 256, nlb = (GRAM_ROWS * cb + 255) / 256;  // <= 5 (<= 3 in FP64)
  C2 ra[5], rb[5];
  auto fetch = [&](int r0) {
#pragma unroll
    for (int u = 0; u < 5; ++u) {
      int t = threadIdx.x + 256 * u;
      ra[u] = mk<R>(0, 0);
      rb[u] = mk<R>(0, 0);
      if (u < nla && t < GRAM_ROWS * ca) {
        int rr = t % GRAM_ROWS, col = t / GRAM_ROWS, r = r0 + rr;
        if (r < r_end) ra[u] = A.p[col / m][kofs + (long long)(col % m) * n3 + r];
      }
      if (u < nlb && t < GRAM_ROWS * cb) {
        int rr = t % GRAM_ROWS, col = t / GRAM_ROWS, r = r0 + rr;
        if (r < r_end) rb[u] = B.p[col / m][kofs + (long long)(col % m) * n3 + r];
      }
    }
  };
  auto stash = [&](int buf) {
#pragma unroll
    for (int u = 0; u < 5; ++u) {
      int t = threadIdx.x + 256 * u;
      if (u < nla && t < GRAM_ROWS * ca) sA[buf][(t % GRAM_ROWS) * GRAM_LD + t / GRAM_ROWS] = ra[u];
      if (u < nlb && t < GRAM_ROWS * cb) sB[buf][(t % GRAM_ROWS) * GRAM_LD + t / GRAM_ROWS] = rb[u];
    }
  };
  CA acc[TILE][TILE];
#pragma unroll
  for (int i = 0; i < TILE; ++i)
#pragma unroll
    for (int j = 0; j < TILE; ++j) acc[i][j] = mk<RA>(0, 0);
  int buf = 0;
  if (r_begin < r_end) {
    fetch(r_begin);
    stash(0);
  }
  __syncthreads();
  for (int r0 = r_begin; r0 < r_end; r0 += GRAM_ROWS) {
    const bool more = r0 + GRAM_ROWS < r_end;
    if (more) fetch(r0 + GRAM_ROWS);
    const C2* a_t = sA[buf];
    const C2* b_t = sB[buf];
#pragma unroll 4
    for (int rr = 0; rr < GRAM_ROWS; ++rr) {
      C2 a[TILE], b[TILE];
#pragma unroll
      for (int i = 0; i < TILE; ++i) { int c = tx + 16 * i; a[i] = c < ca ? a_t[rr * GRAM_LD + c] : mk<R>(0, 0); }
#pragma unroll
      for (int j = 0; j < TILE; ++j) { int c = ty + 16 * j; b[j] = c < cb ? b_t[rr * GRAM_LD + c] : mk<R>(0, 0); }
#pragma unroll
      for (int i = 0; i < TILE; ++i)
#pragma unroll
        for (int j = 0; j < TILE; ++j) cfmac(acc[i][j], mk<RA>(a[i].x, a[i].y), mk<RA>(b[j].x, b[j].y));
    }
    if (more) stash(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
  C2* out = part + ((long long)k * GRAM_SPLIT + split) * ca * cb;
#pragma unroll
  for (int i = 0; i < TILE; ++i)
#pragma unroll
    for (int j = 0; j < TILE; ++j) {
      int a_ = tx + 16 * i, b_ = ty + 16 * j;
      if (a_ < ca && b_ < cb) out[a_ * cb + b_] = mk<R>((R)acc[i][j].x, (R)acc[i][j].y);
    }
}

template <typename R>
__global__ void k_gram_reduce(const typename cplx_t<R>::type* __restrict__ part, int nsplit, int nel, R scale,
                              typename cplx_t<R>::type* __restrict__ G) {
  typedef typename cplx_t<R>::type C2;
  int k = blockIdx.y;
  int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nel) return;
  const C2* p = part + (long long)k * nsplit * nel + e;
  C2 s = mk<R>(0, 0);
  for (int i = 0; i < nsplit; ++i) s = cadd(s, p[(long long)i * nel]);
  G[(long long)k * nel + e] = cscale(s, scale);
}

int launch_gram_reduce_f(const float2* part, int nsplit, int nel, int nk, float scale, float2* G, cudaStream_t s) {
  dim3 g2(cdiv(nel, 256), nk);
  k_gram_reduce<float><<<g2, 256, 0, s>>>(part, nsplit, nel, scale, G);
  PC_LAUNCH_CHECK();
  return PC_OK;
}

template <typename R>
int launch_gram(BlockList<R> A, int na, BlockList<R> B, int nbk, int nk, int m, int n3, R scale,
                typename cplx_t<R>::type* part, typename cplx_t<R>::type* G, cudaStream_t s, int* status) {
  if (na * m > 72 || nbk * m > 72 || na * m > 80) return PC_EINVAL;
  if constexpr (std::is_same<R, float>::value) {
    if (g_tc_tall && status) return launch_gram_tc(A.p, na, B.p, nbk, nk, m, n3, scale, part, GRAM_SPLIT, G, status, s);
  }
  dim3 grid(nk, GRAM_SPLIT);
  // 16 x 16 threads, TILE x TILE outputs each: 2 x 2 covers up to 32 columns per side
  const bool small = na * m <= 32 && nbk * m <= 32;
  if (small) k_gram<R, R, 2><<<grid, 256, 0, s>>>(A, na, B, nbk, m, n3, part);
  else k_gram<R, R, 5><<<grid, 256, 0, s>>>(A, na, B, nbk, m, n3, part);
  PC_LAUNCH_CHECK();
  int nel = na * m * nbk * m;
  dim3 g2(cdiv(nel, 256), nk);
  k_gram_reduce<R><<<g2, 256, 0, s>>>(part, GRAM_SPLIT, nel, scale, G);
  PC_LAUNCH_CHECK();
  return PC_OK;
}
template int launch_gram<double>(BlockList<double>, int, BlockList<double>, int, int, int, int, double, double2*, double2*, cudaStream_t, int*);
template int launch_gram<float>(BlockList<float>, int, BlockList<float>, int, int, int, int, float, float2*, float2*, cudaStream_t, int*);

// ---------------------------------------------------------------------------
// out[t][k][j][r] = (identity_last ? in[t][last][k][j][r] : 0) + sum_b sum_i in[t][b][k][i][r] C[k][b*m+i][j]
// One thread per row r: every row of every output is written by the thread that read it,
// so the output may alias the last input block.
template <typename R, int MOUT, typename RA>
__global__ __launch_bounds__(128) void k_update(UpdateArgs<R> a) {
  typedef typename cplx_t<R>::type C2;
  typedef typename cplx_t<RA>::type CA;
  __shared__ C2 sC[72 * 24];
  const int k = blockIdx.y, t = blockIdx.z;
  const int nsum = a.identity_last ? a.nblk - 1 : a.nblk;
  const int rows = nsum * a.m;
  const C2* Ck = a.C + (long long)k * a.cstride;
  for (int e = threadIdx.x; e < rows * a.mout; e += blockDim.x) {
    int i = e / a.mout, j = e % a.mout;
    sC[e] = Ck[(long long)i * a.cld + j];
  }
  __syncthreads();
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= a.n3) return;
  CA acc[MOUT];
#pragma unroll
  for (int j = 0; j < MOUT; ++j) acc[j] = mk<RA>(0, 0);
  if (a.identity_last) {
    const C2* src = a.in[t][a.nblk - 1] + (long long)k * a.in_kstride + r;
#pragma unroll
    for (int j = 0; j < MOUT; ++j)
      if (j < a.mout) { C2 v = src[(long long)j * a.n3]; acc[j] = mk<RA>(v.x, v.y); }
  }
  for (int b = 0; b < nsum; ++b) {
    const C2* src = a.in[t][b] + (long long)k * a.in_kstride + r;
    for (int i = 0; i < a.m; ++i) {
      C2 v = src[(long long)i * a.n3];
      CA va = mk<RA>(v.x, v.y);
      const C2* crow = sC + (b * a.m + i) * a.mout;
#pragma unroll
      for (int j = 0; j < MOUT; ++j)
        if (j < a.mout) cfma(acc[j], va, mk<RA>(crow[j].x, crow[j].y));
    }
  }
  C2* dst = a.out[t] + (long long)k * a.out_kstride + r;
#pragma unroll
  for (int j = 0; j < MOUT; ++j)
    if (j < a.mout) dst[(long long)j * a.n3] = mk<R>((R)acc[j].x, (R)acc[j].y);
}

template <typename R> static int launch_update_cuda(const UpdateArgs<R>& a, cudaStream_t s) {
  int nsum = a.identity_last ? a.nblk - 1 : a.nblk;
  if (nsum * a.m * a.mout > 72 * 24 || a.mout > 24) return PC_EINVAL;
  dim3 grid(cdiv(a.n3, 128), a.nk, a.ntrip);
  if (a.mout <= 8) k_update<R, 8, R><<<grid, 128, 0, s>>>(a);
  else if (a.mout <= 16) k_update<R, 16, R><<<grid, 128, 0, s>>>(a);
  else k_update<R, 24, R><<<grid, 128, 0, s>>>(a);
  PC_LAUNCH_CHECK();
  return PC_OK;
}

// out[t] = [in] C (and out2[t] = [in] C2nd when a second coefficient set is given).  The CUDA-core
// kernel takes one set per launch; the tensor-core kernel (FP32) takes both in one pass.
template <typename R> int launch_update(const UpdateArgs<R>& a, cudaStream_t s) {
  if constexpr (std::is_same<R, float>::value) {
    if (g_tc_tall && a.status) return launch_update_tc(a, a.status, s);
  }
  int rc = launch_update_cuda<R>(a, s);
  if (rc || !a.C2nd) return rc;
  UpdateArgs<R> b = a;
  b.C = a.C2nd;
  for (int t = 0; t < 3; ++t) b.out[t] = a.out2[t];
  b.C2nd = nullptr;
  return launch_update_cuda<R>(b, s);
}
template int launch_update<double>(const UpdateArgs<double>&, cudaStream_t);
template int launch_update<float>(const UpdateArgs<float>&, cudaStream_t);

// ---------------------------------------------------------------------------
// Cholesky-QR transform: T = D Li^H with zero columns for dropped coordinates.
// One warp factors (warp_chol_inverse); the others only load, scale and store.
template <typename R>
__global__ __launch_bounds__(128) void k_small_chol(const typename cplx_t<R>::type* __restrict__ G, int m, R drop_tol,
                                                    const typename cplx_t<R>::type* __restrict__ Gref, int rows_ref,
                                                    R rel_tol, typename cplx_t<R>::type* __restrict__ T) {
  typedef typename cplx_t<R>::type C2;
  __shared__ C2 B[24 * 25];
  __shared__ C2 X[24 * 25];
  __shared__ R D[24];
  __shared__ int drop[24];
  const int ld = m | 1;
  const int k = blockIdx.x;
  const C2* g = G + (long long)k * m * m;
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    R d = g[i * m + i].x;
    bool keep = (d > (R)0 && d == d);
    if (keep && Gref) {
      R before = -Gref[(long long)k * rows_ref * m + (long long)(rows_ref - m + i) * m + i].x;
      keep = d > rel_tol * before;
    }
    D[i] = keep ? (R)1 / sqrt(d) : (R)0;
    drop[i] = 0;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
    int i = t / m, c = t % m;
    C2 b1 = g[i * m + c], b2 = g[c * m + i];
    R s = D[i] * D[c] * (R)0.5;
    B[i * ld + c] = mk<R>((b1.x + b2.x) * s, (b1.y - b2.y) * s);
  }
  __syncthreads();
  if (threadIdx.x < 32) warp_chol_inverse<R>(B, X, m, ld, drop_tol, drop);
  __syncthreads();
  C2* tk = T + (long long)k * m * m;
  for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
    int i = t / m, c = t % m;
    // T[i][c] = D_i conj(Li[c][i]); dropped columns vanish
    C2 v = (c >= i && !drop[c]) ? cscale(cconj(X[c * ld + i]), D[i]) : mk<R>(0, 0);
    tk[t] = v;
  }
}
template <typename R>
int launch_small_chol(const typename cplx_t<R>::type* G, int m, int nk, R drop_tol,
                      const typename cplx_t<R>::type* Gref, int rows_ref, R rel_tol, typename cplx_t<R>::type* T,
                      cudaStream_t s) {
  if (m > 24) return PC_EINVAL;
  k_small_chol<R><<<nk, 128, 0, s>>>(G, m, drop_tol, Gref, rows_ref, rel_tol, T);
  PC_LAUNCH_CHECK();
  return PC_OK;
}
template int launch_small_chol<double>(const double2*, int, int, double, const double2*, int, double, double2*, cudaStream_t);
template int launch_small_chol<float>(const float2*, int, int, float, const float2*, int, float, float2*, cudaStream_t);

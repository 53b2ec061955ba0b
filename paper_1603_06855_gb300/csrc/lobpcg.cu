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


// FP32 on CUDA cores, the reference of the tensor-core kernel's self-check: G_part[k][split] = A^H B over
// one row range; each of the 16 x 16 threads holds TILE x TILE outputs.  Shared tiles are
// double-buffered: the next tile of GRAM_ROWS rows is fetched into registers while the current one is
// multiplied.
template <int TILE>
__global__ __launch_bounds__(256) void k_gram(BlockList<float> A, int na, BlockList<float> B, int nbk, int m, int n3,
                                              const int* __restrict__ klist, float2* __restrict__ part) {
  typedef float2 C2;
  constexpr int GRAM_ROWS = 16;
  __shared__ C2 sA[2][GRAM_ROWS * GRAM_LD];
  __shared__ C2 sB[2][GRAM_ROWS * GRAM_LD];
  const int k = blockIdx.x, split = blockIdx.y;
  const int ca = na * m, cb = nbk * m;
  const long long kofs = (long long)(klist ? klist[k] : k) * m * n3;
  const int chunk = (n3 + (int)gridDim.y - 1) / (int)gridDim.y;
  const int r_begin = split * chunk, r_end = min(n3, r_begin + chunk);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  // each thread stages elements t = threadIdx.x + 256 u of the (rows x cols) tiles
  const int nla = (GRAM_ROWS * ca + 255) / 256, nlb = (GRAM_ROWS * cb + 255) / 256;  // <= 5
  C2 ra[5], rb[5];
  auto fetch = [&](int r0) {
#pragma unroll
    for (int u = 0; u < 5; ++u) {
      int t = threadIdx.x + 256 * u;
      ra[u] = make_float2(0.f, 0.f);
      rb[u] = make_float2(0.f, 0.f);
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
  C2 acc[TILE][TILE];
#pragma unroll
  for (int i = 0; i < TILE; ++i)
#pragma unroll
    for (int j = 0; j < TILE; ++j) acc[i][j] = make_float2(0.f, 0.f);
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
      for (int i = 0; i < TILE; ++i) { int c = tx + 16 * i; a[i] = c < ca ? a_t[rr * GRAM_LD + c] : make_float2(0.f, 0.f); }
#pragma unroll
      for (int j = 0; j < TILE; ++j) { int c = ty + 16 * j; b[j] = c < cb ? b_t[rr * GRAM_LD + c] : make_float2(0.f, 0.f); }
#pragma unroll
      for (int i = 0; i < TILE; ++i)
#pragma unroll
        for (int j = 0; j < TILE; ++j) cfmac(acc[i][j], a[i], b[j]);
    }
    if (more) stash(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
  C2* out = part + ((long long)k * gridDim.y + split) * ca * cb;
#pragma unroll
  for (int i = 0; i < TILE; ++i)
#pragma unroll
    for (int j = 0; j < TILE; ++j) {
      int a_ = tx + 16 * i, b_ = ty + 16 * j;
      if (a_ < ca && b_ < cb) out[a_ * cb + b_] = acc[i][j];
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

// The FP64 Gram products, bound by the FP64 pipe (two multiply-adds a clock and SM): a thread owns one
// output, the outputs of all column pairs are numbered through so that every lane has one whatever the
// block width (a square tile per thread wasted two thirds of the work at 48 columns), in CTAs of at most
// 608, and the rows are split until some four CTAs per SM share them.  Reference solve (16 x 16 to
// 48 x 48 columns, 375 rows, 4 k): 174 -> 28 us a launch on average.
constexpr int GRAM64_ROWS = 16;
__global__ __launch_bounds__(608) void k_gram64(BlockList<double> A, int na, BlockList<double> B, int nbk, int m, int n3,
                                                int chunk, const int* __restrict__ klist, double2* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char gram_smem[];
  const int ca = na * m, cb = nbk * m;
  const int lda = ca | 1, ldb = cb | 1;
  double2* sA = (double2*)gram_smem;       // GRAM64_ROWS x lda
  double2* sB = sA + GRAM64_ROWS * lda;    // GRAM64_ROWS x ldb
  const int split = blockIdx.y, nsplit = gridDim.y, k = blockIdx.z;
  const long long kofs = (long long)(klist ? klist[k] : k) * m * n3;
  const int r_begin = split * chunk, r_end = min(n3, r_begin + chunk);
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const bool mine = e < ca * cb;
  const int i = mine ? e / cb : 0, j = mine ? e - i * cb : 0;
  double2 acc = make_double2(0.0, 0.0);
  for (int r0 = r_begin; r0 < r_end; r0 += GRAM64_ROWS) {
    for (int t = threadIdx.x; t < GRAM64_ROWS * (ca + cb); t += blockDim.x) {
      const int rr = t % GRAM64_ROWS, c = t / GRAM64_ROWS, r = r0 + rr;
      const bool isA = c < ca;
      const int col = isA ? c : c - ca;
      const double2* src = (isA ? A.p[col / m] : B.p[col / m]) + kofs + (long long)(col % m) * n3;
      const double2 v = r < r_end ? src[r] : make_double2(0.0, 0.0);
      if (isA) sA[rr * lda + col] = v;
      else sB[rr * ldb + col] = v;
    }
    __syncthreads();
#pragma unroll 4
    for (int rr = 0; rr < GRAM64_ROWS; ++rr) cfmac(acc, sA[rr * lda + i], sB[rr * ldb + j]);
    __syncthreads();
  }
  if (mine) part[((long long)k * nsplit + split) * ca * cb + e] = acc;
}

static int launch_gram64(const BlockList<double>& A, int na, const BlockList<double>& B, int nbk, int nk, int m, int n3,
                         double scale, double2* part, int max_split, double2* G, const int* klist, cudaStream_t s) {
  const int nel = na * m * nbk * m;
  const int nx = cdiv(nel, 608);
  const int threads = cdiv(cdiv(nel, nx), 32) * 32;
  int split = 1;
  while (split < max_split && (long long)nx * split * nk < 4LL * device_sms()) ++split;
  const int chunk = cdiv(cdiv(n3, split), GRAM64_ROWS) * GRAM64_ROWS;
  const size_t sm = sizeof(double2) * GRAM64_ROWS * ((size_t)((na * m) | 1) + ((nbk * m) | 1));
  k_gram64<<<dim3(nx, split, nk), threads, sm, s>>>(A, na, B, nbk, m, n3, chunk, klist, part);
  PC_LAUNCH_CHECK();
  dim3 g2(cdiv(nel, 256), nk);
  k_gram_reduce<double><<<g2, 256, 0, s>>>(part, split, nel, scale, G);
  PC_LAUNCH_CHECK();
  return PC_OK;
}

template <typename R>
int launch_gram(BlockList<R> A, int na, BlockList<R> B, int nbk, int nk, int m, int n3, R scale,
                typename cplx_t<R>::type* part, typename cplx_t<R>::type* G, MatRef<R>* out, cudaStream_t s, int* status,
                const int* klist, int max_split) {
  if (na * m > 72 || nbk * m > 72 || max_split < 1 || max_split > GRAM_SPLIT) return PC_EINVAL;
  const int nel = na * m * nbk * m;
  if constexpr (std::is_same<R, float>::value) {
    if (g_tc_tall && status)
      return launch_gram_tc(A.p, na, B.p, nbk, nk, m, n3, scale, part, max_split, out, status, klist, s);
  }
  *out = MatRef<R>();
  out->p = G;
  out->nel = nel;
  if constexpr (std::is_same<R, double>::value) {
    return launch_gram64(A, na, B, nbk, nk, m, n3, scale, part, max_split, G, klist, s);
  } else {
    dim3 grid(nk, max_split);
    // 16 x 16 threads, TILE x TILE outputs each: 2 x 2 covers up to 32 columns per side
    const bool small = na * m <= 32 && nbk * m <= 32;
    if (small) k_gram<2><<<grid, 256, 0, s>>>(A, na, B, nbk, m, n3, klist, part);
    else k_gram<5><<<grid, 256, 0, s>>>(A, na, B, nbk, m, n3, klist, part);
    PC_LAUNCH_CHECK();
    return launch_gram_reduce_f(part, max_split, nel, nk, scale, G, s);
  }
}
template int launch_gram<double>(BlockList<double>, int, BlockList<double>, int, int, int, int, double, double2*, double2*, MatRef<double>*, cudaStream_t, int*, const int*, int);
template int launch_gram<float>(BlockList<float>, int, BlockList<float>, int, int, int, int, float, float2*, float2*, MatRef<float>*, cudaStream_t, int*, const int*, int);

// ---------------------------------------------------------------------------
// out[t][k][j][r] = (identity_last ? in[t][last][k][j][r] : 0) + sum_b sum_i in[t][b][k][i][r] C[k][b*m+i][j]
// One thread per row r: every row of every output is written by the thread that read it,
// so the output may alias the last input block.
template <int MOUT>
__global__ __launch_bounds__(128) void k_update(UpdateArgs<float> a) {
  typedef float2 C2;
  __shared__ C2 sC[72 * 24];
  const int k = a.klist ? a.klist[blockIdx.y] : (int)blockIdx.y, t = blockIdx.z;
  const int nsum = a.identity_last ? a.nblk - 1 : a.nblk;
  const int rows = nsum * a.m;
  for (int e = threadIdx.x; e < rows * a.mout; e += blockDim.x) {
    int i = e / a.mout, j = e % a.mout;
    sC[e] = a.C.at(blockIdx.y, i * a.cld + j);
  }
  __syncthreads();
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= a.n3) return;
  C2 acc[MOUT];
#pragma unroll
  for (int j = 0; j < MOUT; ++j) acc[j] = make_float2(0.f, 0.f);
  if (a.identity_last) {
    const C2* src = a.in[t][a.nblk - 1] + (long long)k * a.in_kstride + r;
#pragma unroll
    for (int j = 0; j < MOUT; ++j)
      if (j < a.mout) { C2 v = src[(long long)j * a.n3]; acc[j] = v; }
  }
  for (int b = 0; b < nsum; ++b) {
    const C2* src = a.in[t][b] + (long long)k * a.in_kstride + r;
    for (int i = 0; i < a.m; ++i) {
      C2 v = src[(long long)i * a.n3];
      const C2* crow = sC + (b * a.m + i) * a.mout;
#pragma unroll
      for (int j = 0; j < MOUT; ++j)
        if (j < a.mout) cfma(acc[j], v, crow[j]);
    }
  }
  C2* dst = a.out[t] + (long long)k * a.out_kstride + r;
#pragma unroll
  for (int j = 0; j < MOUT; ++j)
    if (j < a.mout) dst[(long long)j * a.n3] = acc[j];
}

// FP64 updates: 32 rows of all outputs per CTA, a warp per group of JT outputs (one row per lane), so
// that small problems fill the chip (a reference solve, 375 rows, 16 outputs, 4 k: 36 CTAs -> 144) and
// the FP64 pipe, which is the bound, has up to eight warps' independent sums to draw on.  All inputs of a CTA's
// rows are read before any output is written, so the output may alias an input block.  Reference solve
// 82 -> 22 us a launch; final step (2187 rows, 23 outputs, 50 k, three triplets) 804 -> 671 us.
template <int JT>
__global__ __launch_bounds__(256) void k_update64(UpdateArgs<double> a) {
  __shared__ double2 sC[72 * 24];
  const int k = a.klist ? a.klist[blockIdx.y] : (int)blockIdx.y, t = blockIdx.z;
  const int nsum = a.identity_last ? a.nblk - 1 : a.nblk;
  const int rows = nsum * a.m;
  for (int e = threadIdx.x; e < rows * 24; e += blockDim.x) {
    const int i = e / 24, j = e % 24;
    sC[e] = j < a.mout ? a.C.at(blockIdx.y, i * a.cld + j) : make_double2(0.0, 0.0);
  }
  __syncthreads();
  const int r = blockIdx.x * 32 + (threadIdx.x & 31);
  const int j0 = (threadIdx.x >> 5) * JT;
  double2 acc[JT];
#pragma unroll
  for (int j = 0; j < JT; ++j) acc[j] = make_double2(0.0, 0.0);
  if (r < a.n3) {
    if (a.identity_last) {
      const double2* src = a.in[t][a.nblk - 1] + (long long)k * a.in_kstride + r;
#pragma unroll
      for (int j = 0; j < JT; ++j)
        if (j0 + j < a.mout) acc[j] = src[(long long)(j0 + j) * a.n3];
    }
    for (int b = 0; b < nsum; ++b) {
      const double2* src = a.in[t][b] + (long long)k * a.in_kstride + r;
#pragma unroll 4
      for (int i = 0; i < a.m; ++i) {
        const double2 v = src[(long long)i * a.n3];
        const double2* crow = sC + (b * a.m + i) * 24 + j0;
#pragma unroll
        for (int j = 0; j < JT; ++j) cfma(acc[j], v, crow[j]);
      }
    }
  }
  __syncthreads();
  if (r >= a.n3) return;
  double2* dst = a.out[t] + (long long)k * a.out_kstride + r;
#pragma unroll
  for (int j = 0; j < JT; ++j)
    if (j0 + j < a.mout) dst[(long long)(j0 + j) * a.n3] = acc[j];
}

template <typename R> static int launch_update_cuda(const UpdateArgs<R>& a, cudaStream_t s) {
  int nsum = a.identity_last ? a.nblk - 1 : a.nblk;
  if (nsum * a.m * a.mout > 72 * 24 || a.mout > 24) return PC_EINVAL;
  if constexpr (std::is_same<R, double>::value) {
    const dim3 grid(cdiv(a.n3, 32), a.nk, a.ntrip);
    if (a.mout <= 8) k_update64<1><<<grid, 32 * a.mout, 0, s>>>(a);
    else if (a.mout <= 16) k_update64<2><<<grid, 32 * cdiv(a.mout, 2), 0, s>>>(a);
    else k_update64<3><<<grid, 32 * cdiv(a.mout, 3), 0, s>>>(a);
  } else {
    const dim3 grid(cdiv(a.n3, 128), a.nk, a.ntrip);
    if (a.mout <= 8) k_update<8><<<grid, 128, 0, s>>>(a);
    else if (a.mout <= 16) k_update<16><<<grid, 128, 0, s>>>(a);
    else k_update<24><<<grid, 128, 0, s>>>(a);
  }
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
  if (rc || !a.C2nd.p) return rc;
  UpdateArgs<R> b = a;
  b.C = a.C2nd;
  for (int t = 0; t < 3; ++t) b.out[t] = a.out2[t];
  b.C2nd.p = nullptr;
  return launch_update_cuda<R>(b, s);
}
template int launch_update<double>(const UpdateArgs<double>&, cudaStream_t);
template int launch_update<float>(const UpdateArgs<float>&, cudaStream_t);

// ---------------------------------------------------------------------------
// Cholesky-QR transform: T = D Li^H with zero columns for dropped coordinates.
// One warp factors (warp_chol_inverse); the others only load, scale and store.
template <typename R>
__global__ __launch_bounds__(128) void k_small_chol(MatRef<R> G, int m, R drop_tol, typename cplx_t<R>::type* __restrict__ T) {
  typedef typename cplx_t<R>::type C2;
  __shared__ C2 B[24 * 25];
  __shared__ C2 X[24 * 25];
  __shared__ R D[24];
  __shared__ int drop[24];
  const int ld = m | 1;
  const int k = blockIdx.x;
  for (int t = threadIdx.x; t < m * m; t += blockDim.x) X[(t / m) * ld + t % m] = G.at(k, t);
  __syncthreads();
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    const R d = X[i * ld + i].x;
    D[i] = (d > (R)0 && d == d) ? (R)1 / sqrt(d) : (R)0;
    drop[i] = 0;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
    int i = t / m, c = t % m;
    const C2 b1 = X[i * ld + c], b2 = X[c * ld + i];
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
int launch_small_chol(const MatRef<R>& G, int m, int nk, R drop_tol, typename cplx_t<R>::type* T, cudaStream_t s) {
  if (m > 24) return PC_EINVAL;
  k_small_chol<R><<<nk, 128, 0, s>>>(G, m, drop_tol, T);
  PC_LAUNCH_CHECK();
  return PC_OK;
}
template int launch_small_chol<double>(const MatRef<double>&, int, int, double, double2*, cudaStream_t);
template int launch_small_chol<float>(const MatRef<float>&, int, int, float, float2*, cudaStream_t);

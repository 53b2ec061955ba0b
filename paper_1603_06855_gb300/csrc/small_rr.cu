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
//     CTA (pdir: Cholesky-QR of the part of the old Ritz block outside the new one).
// Bound: the chain of a Jacobi round (barrier, plane loads, rotated entry, new plane: 740 of 970
// cycles at n = 57) for small n, issue and shared-memory bandwidth of one SM for n near 72.  50
// problems of the design workloads: n = 45 400 -> 170 us, n = 57 583 -> 238-269 us, n = 69 885 -> 372 us
// against positions that moved by index tables, V accumulated beside the rotations (its traffic was
// 60 % of the rounds' shared-memory bytes) and CTA-wide barriers in every column of the reductions.
// This is the mixed form's version (FP32, four 72 x 74 complex matrices in shared memory);
// FP64 problems have theirs (small_rr64.cu).
#include <algorithm>
#include "jacobi.cuh"

namespace {
constexpr int SR_THREADS = 1024;
constexpr int SR_PB = 8;  // panel / row-block width of the reductions
}  // namespace

__global__ __launch_bounds__(SR_THREADS) void k_small_rr32(MatRef<float> GA, MatRef<float> GO, int n, int m,
                                                          float drop_tol, const int* __restrict__ klist,
                                                         float* __restrict__ lam_out, float2* __restrict__ coef,
                                                         float2* __restrict__ cpo, float pdir_abs, int* status,
                                                         double* flops, unsigned char* scratch, long long stride) {
  extern __shared__ __align__(16) unsigned char smem[];
  float2* B0 = (float2*)smem;          // GO -> L -> Jacobi buffer 1
  float2* B1 = B0 + SR_MAT;            // GA -> T = L^-1 GA -> Jacobi buffer 0
  float2* Vt = B1 + SR_MAT;            // L^-1
  float2* Cm = Vt + SR_MAT;            // C = L^-1 GA L^-H (original order) -> Y
  Plane<float>* pl = (Plane<float>*)(Cm + SR_MAT);   // 2 x 36 planes (by round parity)
  float* D = (float*)(pl + 2 * 36);    // SR_NMAX
  float* ev = D + SR_NMAX;             // SR_NMAX: reciprocal diagonal of L, then eigenvalues
  int* drop = (int*)(ev + SR_NMAX);    // SR_NMAX
  int* idx = drop + SR_NMAX;           // SR_NMAX: position -> coordinate (-1: padding)
  int* perm = idx + SR_NMAX;           // SR_NMAX
  int* low = perm + SR_NMAX;           // SR_NMAX: among the m smallest diagonal entries
  int* misc = low + SR_NMAX;           // [0] kept count, [2] floor bits, [3] sweeps
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int k = blockIdx.x;                        // problem
  const int kp = klist ? klist[k] : k;             // its k-point
  Plane<float>* logk = (Plane<float>*)(scratch + k * stride);  // rotations of this problem, np planes per round
  float2* ck = coef + (long long)k * n * m;
  float2* cpk = cpo ? cpo + (long long)k * n * m : nullptr;  // conjugate-direction coefficients (or none)
  // 1. scaling, symmetrised copies, identity right-hand side of L^-1 (in Vt)
  for (int i = warp; i < n; i += 32)
    for (int c = lane; c < n; c += 32) {
      B1[i * SR_LD + c] = GA.at(k, i * n + c);
      B0[i * SR_LD + c] = GO.at(k, i * n + c);
      Vt[i * SR_LD + c] = make_float2(i == c ? 1.f : 0.f, 0.f);
    }
  __syncthreads();
  for (int i = tid; i < n; i += blockDim.x) {
    const float d = B0[i * SR_LD + i].x;
    D[i] = (d > 0.f && d == d) ? 1.f / sqrtf(d) : 0.f;
    drop[i] = 0;
  }
  __syncthreads();
  for (int i = warp; i < n; i += 32)
    for (int c = i + lane; c < n; c += 32) {  // this thread alone reads and writes (i, c) and (c, i)
      const float2 a1 = B1[i * SR_LD + c], a2 = B1[c * SR_LD + i];
      const float2 b1 = B0[i * SR_LD + c], b2 = B0[c * SR_LD + i];
      const float s = D[i] * D[c] * 0.5f;
      const float2 a = make_float2((a1.x + a2.x) * s, (a1.y - a2.y) * s), b = make_float2((b1.x + b2.x) * s, (b1.y - b2.y) * s);
      B1[i * SR_LD + c] = a;
      B0[i * SR_LD + c] = b;
      if (c > i) {
        B1[c * SR_LD + i] = cconj(a);
        B0[c * SR_LD + i] = cconj(b);
      }
    }
  __syncthreads();
  // 2. Cholesky of B0 (lower)
  block_cholesky<float, SR_PB, SR_THREADS>(B0, n, drop_tol, drop, ev);
  // 3. T = L^-1 GA (in place in B1) and L^-1 (in place in Vt), then C = L^-1 T^H in Cm (upper)
  block_forward<float, SR_PB, SR_THREADS>(B0, ev, B1, Vt, n, n, 2 * n, 1);
  for (int i = warp; i < n; i += 32)
    for (int j = lane; j < n; j += 32) Cm[i * SR_LD + j] = cconj(B1[j * SR_LD + i]);
  __syncthreads();
  block_forward<float, SR_PB, SR_THREADS>(B0, ev, Cm, (float2*)nullptr, n, n, n, 2);
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
    for (int j = tid; j < m; j += blockDim.x) lam_out[(long long)kp * m + j] = GA.at(k, j * n + j).x / GO.at(k, j * n + j).x;
    if (tid == 0) set_status(status, PC_ENOCONV);
    if (cpk) {
      for (int t = tid; t < n * m; t += blockDim.x) {
        const int i = t / m, j = t % m;
        B1[t] = make_float2(i == j ? 1.f : 0.f, 0.f);
      }
      __syncthreads();
      pdir<float, SR_THREADS>(GO, k, n, m, pdir_abs, B0, B1, B1 + n * m, B1 + 2 * n * m, Cm, Cm + m * (m | 1), ev, drop, cpk);
    }
    return;
  }
  const int npad = nk_ + (nk_ & 1), np = npad / 2, nrounds = npad - 1;
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
  const int sweeps = jacobi_sweeps<float, SR_THREADS>(B1, B0, pl, logk, nk_, m, floor_abs, true, ev, perm, low, misc);
  // 5. lowest m eigenpairs of the kept coordinates
  // eigenvectors of the packed matrix for these m: the logged rotations, last round first
  float2* Y = Cm;  // nk_ x m
  const int K = sweeps * nrounds;
  const float2* Sf = (K & 1) ? B0 : B1;
  Plane<float>*c0 = (Plane<float>*)B1, *c1 = (Plane<float>*)B0;
  if (np <= 16) replay<float, 16, 1, SR_THREADS>(logk, K, np, nk_, m, perm, c0, c1, Y, m, Sf, ev);
  else if (np <= 32) replay<float, 16, 2, SR_THREADS>(logk, K, np, nk_, m, perm, c0, c1, Y, m, Sf, ev);
  else replay<float, 16, 3, SR_THREADS>(logk, K, np, nk_, m, perm, c0, c1, Y, m, Sf, ev);
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
  for (int j = tid; j < m; j += blockDim.x) lam_out[(long long)kp * m + j] = ev[perm[j]];
  if (cpk) {
    __syncthreads();
    pdir<float, SR_THREADS>(GO, k, n, m, pdir_abs, B0, B1, B1 + n * m, B1 + 2 * n * m, Cm, Cm + m * (m | 1), ev, drop, cpk);
  }
  if (flops && tid == 0) {
    // algorithmic work: Cholesky n^3/6, L^-1 GA n^3/2, L^-1 T^H n^3/2 and L^-1 n^3/6 complex
    // multiply-adds (8 real flops each); per Jacobi sweep n_k (n_k - 1) / 2 rotations, each
    // updating 2 n_k entries of C and 2 n entries of V at 12 real flops per entry
    const double nn = n, kk = nk_;
    atomicAdd(flops, 8.0 * (4.0 / 3.0) * nn * nn * nn + sweeps * kk * (kk - 1.0) * 0.5 * 24.0 * (kk + nn));
  }
}

// Planes (16 bytes) of the rotations of the most sweeps and of the round after them.
long long small_rr32_scratch(int n) { return 16LL * ((long long)SR_MAX_SWEEPS * n + 1) * ((n + 1) / 2); }

int launch_small_rr32(const MatRef<float>& GA, const MatRef<float>& GO, int n, int m, int nk, float drop_tol, const int* klist,
                      float* lam_out, float2* coef, float2* cp, float pdir_abs, int* status, double* flops,
                      void* scratch, long long stride, int slots, cudaStream_t s) {
  if (n > SR_NMAX || m > n || m > 24 || n < 1 || slots < 1 || stride < small_rr32_scratch(n) || stride % 16) return PC_EINVAL;
  const size_t sm = sizeof(float2) * 4 * (size_t)SR_MAT + sizeof(Plane<float>) * 72 + sizeof(float) * 2 * SR_NMAX +
                    sizeof(int) * (4 * SR_NMAX + 8);
  static const cudaError_t attr =  // once, thread-safe (k groups launch from several host threads)
      cudaFuncSetAttribute(k_small_rr32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  (void)attr;
  for (int f = 0; f < nk; f += slots) {
    const long long o = (long long)f * n * m;
    k_small_rr32<<<std::min(slots, nk - f), SR_THREADS, sm, s>>>(
        GA.from(f), GO.from(f), n, m, drop_tol, klist ? klist + f : nullptr, klist ? lam_out : lam_out + (long long)f * m,
        coef + o, cp ? cp + o : nullptr, pdir_abs, status, flops, (unsigned char*)scratch, stride);
    PC_LAUNCH_CHECK();
  }
  return PC_OK;
}

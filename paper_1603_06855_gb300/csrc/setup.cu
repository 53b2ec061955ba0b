// Per-design operator assembly (k-independent):
//   SIMP interpolation           -- Methods, eq. combinematerial (linear in chi = rho^p)
//   structure factors            -- Methods, eq. loop: centroid sums of the fields times
//                                   exp(i 2 pi Delta.s_e) for every plane-wave difference Delta
//   Toeplitz operators           -- Results, eqs. intOmega / intPhi via eq. matrixofintegral:
//                                   T_c[p][q] = V c^(g_q - g_p)
//   inverse compliance operators -- the stress elimination of eq. matrixform; both phases are
//                                   isotropic, so Phi^-1 only needs the inverses of the bulk
//                                   (f1 = (1-2nu)/E) and shear (f2 = (1+nu)/E) Toeplitz blocks.
#include "kernels.h"
#include "small_dense.cuh"

// ---------------------------------------------------------------------------
// SIMP interpolation: fields[0] = density, fields[1] = f1, fields[2] = f2 per element, and
// dfc = (d f1 / d chi, d f2 / d chi) per element (dfc may be NULL).  PC_LAW_COMPLIANCE: f1, f2
// linear in chi; PC_LAW_YOUNG: E and nu linear in chi, f1 = (1 - 2 nu)/E, f2 = (1 + nu)/E, so
// d f1/d chi = (-2 dnu E - (1 - 2 nu) dE) / E^2 and d f2/d chi = (dnu E - (1 + nu) dE) / E^2.
__global__ void k_interp(const double* __restrict__ rho, int ne, MaterialConsts mc,
                         double* __restrict__ fields, double* __restrict__ dchi,
                         double* __restrict__ chi_out, int* status, double* __restrict__ dfc) {
  int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= ne) return;
  double r = rho[e];
  if (!(r >= 0.0 && r <= 1.0)) {  // also catches NaN
    set_status(status, PC_EDOMAIN);
    r = (r > 1.0) ? 1.0 : 0.0;
    if (!(rho[e] == rho[e])) r = 0.0;
  }
  double chi, dc;
  if (mc.penal == 1.0) { chi = r; dc = 1.0; }
  else { chi = pow(r, mc.penal); dc = (r > 0.0) ? mc.penal * pow(r, mc.penal - 1.0) : 0.0; }
  fields[e] = mc.rho0 + chi * (mc.rho1 - mc.rho0);
  double f1, f2, d1, d2;
  if (mc.law == PC_LAW_YOUNG) {
    const double dE = mc.E1 - mc.E0, dn = mc.nu1 - mc.nu0;
    const double E = mc.E0 + chi * dE, nu = mc.nu0 + chi * dn;
    f1 = (1.0 - 2.0 * nu) / E;
    f2 = (1.0 + nu) / E;
    d1 = (-2.0 * dn * E - (1.0 - 2.0 * nu) * dE) / (E * E);
    d2 = (dn * E - (1.0 + nu) * dE) / (E * E);
  } else {
    f1 = mc.f1_0 + chi * (mc.f1_1 - mc.f1_0);
    f2 = mc.f2_0 + chi * (mc.f2_1 - mc.f2_0);
    d1 = mc.f1_1 - mc.f1_0;
    d2 = mc.f2_1 - mc.f2_0;
  }
  fields[ne + e] = f1;
  fields[2 * ne + e] = f2;
  if (dfc) {
    dfc[e] = d1;
    dfc[ne + e] = d2;
  }
  dchi[e] = dc;
  chi_out[e] = chi;
}

// Mean of chi (deterministic single-block reduction) for the preconditioner's reference medium.
__global__ void k_mean(const double* __restrict__ x, int n, double* out) {
  __shared__ double red[1024];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += x[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0] / (double)n;
}

// Structure factors by three separable sums, one grid axis at a time.  The phases of an axis of n
// voxels, exp(i pi D (2j+1)/n), take only 2n values: a CTA tabulates them in shared memory (8 KB at
// most) and steps through the table, two or four FP64 multiply-adds a term instead of a sine and a cosine
// (32^3 voxels, M = 4: 460 -> 37 us for the three stages, the same bits).
#define SFAC_NMAX 256
__device__ __forceinline__ void phase_table(double2* tab, int n) {
  for (int t = threadIdx.x; t < 2 * n; t += blockDim.x) tab[t] = phase_pi_over(t, n);
  __syncthreads();
}
// Stage 1 (axis 2): t1[f][i][j][d3] = sum_l c_f[i][j][l] exp(i pi D3 (2l+1)/n2), D3 = d3 - 2M.
__global__ void k_sfac1(const double* __restrict__ fields, int n0, int n1, int n2, int M,
                        double2* __restrict__ t1) {
  __shared__ double2 tab[2 * SFAC_NMAX];
  phase_table(tab, n2);
  int L = 4 * M + 1;
  long long total = 3LL * n0 * n1 * L;
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= total) return;
  int d3 = (int)(t % L);
  long long r = t / L;           // (f, i, j)
  const int D = (((d3 - 2 * M) % (2 * n2)) + 2 * n2) % (2 * n2);  // phase index of l = 0, its step is 2 D
  const int step = (2 * D) % (2 * n2);
  const double* src = fields + r * n2;
  double2 acc = make_double2(0.0, 0.0);
  for (int l = 0, q = D; l < n2; ++l) {
    const double2 ph = tab[q];
    acc.x = fma(src[l], ph.x, acc.x);
    acc.y = fma(src[l], ph.y, acc.y);
    q += step;
    q -= q >= 2 * n2 ? 2 * n2 : 0;
  }
  t1[t] = acc;
}
// Stage 2 (axis 1): t2[f][i][d2][d3] = sum_j t1[f][i][j][d3] exp(i pi D2 (2j+1)/n1).
__global__ void k_sfac2(const double2* __restrict__ t1, int n0, int n1, int M, double2* __restrict__ t2) {
  __shared__ double2 tab[2 * SFAC_NMAX];
  phase_table(tab, n1);
  int L = 4 * M + 1;
  long long total = 3LL * n0 * L * L;
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= total) return;
  int d3 = (int)(t % L);
  int d2 = (int)((t / L) % L);
  long long fi = t / ((long long)L * L);
  const int D = (((d2 - 2 * M) % (2 * n1)) + 2 * n1) % (2 * n1), step = (2 * D) % (2 * n1);
  double2 acc = make_double2(0.0, 0.0);
  for (int j = 0, q = D; j < n1; ++j) {
    cfma(acc, t1[(fi * n1 + j) * L + d3], tab[q]);
    q += step;
    q -= q >= 2 * n1 ? 2 * n1 : 0;
  }
  t2[t] = acc;
}
// Stage 3 (axis 0): sfac[f][d1][d2][d3] = (1/ne) sum_i t2[f][i][d2][d3] exp(i pi D1 (2i+1)/n0).
__global__ void k_sfac3(const double2* __restrict__ t2, int n0, int M, double inv_ne, double2* __restrict__ sf) {
  __shared__ double2 tab[2 * SFAC_NMAX];
  phase_table(tab, n0);
  int L = 4 * M + 1;
  long long L2 = (long long)L * L;
  long long total = 3LL * L * L2;
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= total) return;
  long long d23 = t % L2;
  int d1 = (int)((t / L2) % L);
  int f = (int)(t / (L2 * L));
  const int D = (((d1 - 2 * M) % (2 * n0)) + 2 * n0) % (2 * n0), step = (2 * D) % (2 * n0);
  double2 acc = make_double2(0.0, 0.0);
  for (int i = 0, q = D; i < n0; ++i) {
    cfma(acc, t2[((long long)f * n0 + i) * L2 + d23], tab[q]);
    q += step;
    q -= q >= 2 * n0 ? 2 * n0 : 0;
  }
  sf[t] = cscale(acc, inv_ne);
}

// Toeplitz operators T_f[p][q] = V * c^_f(g_q - g_p), f in {density, f1, f2}, SI units.
__global__ void k_toeplitz(const double2* __restrict__ sf, int M, double V, double2* __restrict__ T) {
  int M2 = 2 * M + 1, N = M2 * M2 * M2, L = 4 * M + 1;
  long long NN = (long long)N * N;
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 3 * NN) return;
  int f = (int)(t / NN);
  long long pq = t % NN;
  int p = (int)(pq / N), q = (int)(pq % N);
  int p1 = p / (M2 * M2), p2 = (p / M2) % M2, p3 = p % M2;
  int q1 = q / (M2 * M2), q2 = (q / M2) % M2, q3 = q % M2;
  int d1 = q1 - p1 + 2 * M, d2 = q2 - p2 + 2 * M, d3 = q3 - p3 + 2 * M;
  double2 v = sf[(long long)f * L * L * L + ((long long)d1 * L + d2) * L + d3];
  T[t] = cscale(v, V);
}

// In-place blocked Gauss-Jordan inversion of Hermitian positive definite matrices (no pivoting is
// needed), on the upper triangle.  With the pivot block 1, P = A11^-1 and R = A1: (its rows), one panel step
// is
//   A11 <- P,   A1j <- (P R)_j,   Ai1 <- -Ai1 P,   Aij <- Aij - Ai1 (P R)_j   (i, j outside the block).
// Rows already swept (i before the block) and those to come keep A_ij = -A_ji^H between them and
// A_ij = A_ji^H among themselves, so the upper triangle of 16 x 16 tiles is enough: R_j = -A_j1^H for a
// swept j, Ai1 = s_i R_i^H with s_i = -1 for a swept i and +1 else, and Ai1 <- ((P R)_i)^H above the block.
// The pivot block enters by the inverse of its Cholesky factor, A11 = L L^H: with Y = L^-1 R the update is
// Aij <- Aij - s_i Y_i^H Y_j, and P R = L^-H Y, P = L^-H L^-1.  An inverse P itself, formed from the block and
// multiplied in, stands for a block that differs by eps cond(A11) of its size, which the condition then
// multiplies once more: T W - 1 of compliance operators of N = 343 and condition 1.7e4 is 8e-12 by the factor,
// 1e-11 to 1e-9 by P, 6e-11 to 2e-6 by P on the whole matrix in 32 columns, and was 2e-7 to 7e-3 by P of a block
// whose two triangles had drifted apart by rounding (everything is taken from upper triangles).
// Two launches a panel: Y, and the update of the tiles (one 16^3 product each, the pivot's rows and columns
// among them), in which one more CTA per matrix factors the next pivot block.  That block is ready early: the update before stored it as of then, and the CTA
// applies this panel's term itself.  The tiles of the next panel's rows store R for the next step.
// blockIdx.z or .y selects the matrix.
//
// Bound: FP64 multiply-adds, 4 N^3 per matrix for the half (N = 729, two matrices: 2.5 ms); 16 columns a
// panel keep the next pivot's chain (16 dependent steps on one SM, some 20 us) beside the update (30 us a
// panel at N = 343, 72 at 729, 200 at 1331).  Both matrices, against the whole matrix with 32 columns a panel,
// three to four launches and two events between streams: N = 343 2.7 -> 0.75 ms, 729 7.6 -> 3.6, 1331 33 -> 18.3.
// P R in the panel launch instead of the pivot's tiles, which would else only copy it: 0.12, 0.2 and 0.4 ms more.
constexpr int GJ_B = 16;
struct GjBufs {
  double2* A;   // 2 x N x N
  double2* R;   // 2 parities x 2 x GJ_B x N: rows of the pivot block
  double2* Y;   // 2 x GJ_B x N: L^-1 R
  double2* Li;  // 2 parities x 2 x GJ_B x GJ_B: L^-1
  double2* D;   // 2 parities x 2 x GJ_B x GJ_B: diagonal blocks two panels ahead
};

// L^-1 of the Hermitian positive definite block held by 256 threads, one entry each (rows and columns past N: the
// identity), from its upper triangle: Gaussian elimination of the block, its row operations applied to the identity,
// whose part below the diagonal takes the place of the lower triangle; then the rows over the roots of the
// pivots.  Every warp forms the pivot's reciprocal for itself (a broadcast would cost a barrier), so it is kept to a
// few FP64 instructions.
__device__ __forceinline__ double2 gj_factor_inverse(double2 v, double2 (*S)[GJ_B + 1]) {
  const int r = threadIdx.x >> 4, c = threadIdx.x & 15;
  if (r > c) v = make_double2(0.0, 0.0);
  for (int k = 0; k < GJ_B; ++k) {
    S[r][c] = v;
    __syncthreads();
    const double ip = inv_newton(S[k][k].x);
    const double2 row = S[k][c], l = cscale(cconj(S[k][r]), -ip);
    if (r > k) {
      if (c == k) v = l;
      else if (c >= r || c < k) cfma(v, l, row);
    }
    __syncthreads();
  }
  S[r][c] = v;
  __syncthreads();
  const double d = inv_sqrt(S[r][r].x);
  return r < c ? make_double2(0.0, 0.0) : (r == c ? make_double2(d, 0.0) : cscale(v, d));
}

// Start: R of panel 0, the factor of pivot block 0 and the diagonal block of panel 1.
__global__ __launch_bounds__(256) void k_gj_start(GjBufs g, int N) {
  __shared__ double2 S[GJ_B][GJ_B + 1];
  const int z = blockIdx.y;
  const double2* A = g.A + (long long)z * N * N;
  const int r = threadIdx.x >> 4, c = threadIdx.x & 15;
  if (blockIdx.x == 0) {
    double2 v = make_double2(r == c ? 1.0 : 0.0, 0.0);
    if (r < N && c < N) v = A[(long long)r * N + c];
    g.Li[z * GJ_B * GJ_B + threadIdx.x] = gj_factor_inverse(v, S);
    const int r1 = GJ_B + r, c1 = GJ_B + c;
    g.D[2 * GJ_B * GJ_B + z * GJ_B * GJ_B + threadIdx.x] =
        (r1 < N && c1 < N) ? A[(long long)r1 * N + c1] : make_double2(r == c ? 1.0 : 0.0, 0.0);
  }
  const int j = blockIdx.x * GJ_B + c;
  if (j < N) g.R[((long long)z * GJ_B + r) * N + j] = r < N ? A[(long long)r * N + j] : make_double2(0.0, 0.0);
}

// Y of one panel (L^-1 is lower triangular; a warp holds rows r and r | 1).
__global__ __launch_bounds__(256) void k_gj_panel(GjBufs g, int N, int par) {
  __shared__ double2 Ls[GJ_B][GJ_B + 1], Rs[GJ_B][GJ_B + 1];
  const int z = blockIdx.y, r = threadIdx.x >> 4, c = threadIdx.x & 15, j = blockIdx.x * GJ_B + c;
  const long long o = ((long long)z * GJ_B + r) * N + j;
  Ls[r][c] = g.Li[(2 * par + z) * GJ_B * GJ_B + threadIdx.x];
  Rs[r][c] = j < N ? g.R[(long long)par * 2 * GJ_B * N + o] : make_double2(0.0, 0.0);
  __syncthreads();
  double2 y = make_double2(0.0, 0.0);
#pragma unroll 2
  for (int l = 0; l <= (r | 1); ++l) cfma(y, Ls[r][l], Rs[l][c]);
  if (j < N) g.Y[o] = y;
}

// One panel step: the upper tiles (blockIdx.x - 1 numbers them by rows), and in blockIdx.x = 0 the next
// pivot block's factor.
__global__ __launch_bounds__(256) void k_gj_update(GjBufs g, int N, int p, int nt) {
  __shared__ double2 X[GJ_B][GJ_B + 1], Z[GJ_B][GJ_B + 1];
  const int z = blockIdx.y, par = p & 1, r = threadIdx.x >> 4, c = threadIdx.x & 15;
  double2* A = g.A + (long long)z * N * N;
  const double2* Y = g.Y + (long long)z * GJ_B * N;
  double2* Rn = g.R + (long long)(2 * (par ^ 1) + z) * GJ_B * N;
  const double2* Li = g.Li + (2 * par + z) * GJ_B * GJ_B;
  const double2 zero = make_double2(0.0, 0.0);
  if (blockIdx.x == 0) {
    if (p + 1 >= nt) return;
    const int j = (p + 1) * GJ_B + c;
    X[r][c] = j < N ? Y[(long long)r * N + j] : zero;
    double2 v = g.D[(2 * (par ^ 1) + z) * GJ_B * GJ_B + threadIdx.x];
    __syncthreads();
    double2 acc = zero;
#pragma unroll
    for (int l = 0; l < GJ_B; ++l) cfmac(acc, X[l][r], X[l][c]);
    v = csub(v, acc);
    __syncthreads();
    g.Li[(2 * (par ^ 1) + z) * GJ_B * GJ_B + threadIdx.x] = gj_factor_inverse(v, X);
    return;
  }
  // tile (I, J), I <= J, number t = I nt - I (I - 1) / 2 + J - I
  const int t = blockIdx.x - 1;
  int I = (int)((2 * nt + 1 - sqrtf((float)(2 * nt + 1) * (2 * nt + 1) - 8.f * t)) * 0.5f);
  I = max(0, min(I, nt - 1));
  while (I > 0 && t < I * nt - I * (I - 1) / 2) --I;
  while (I + 1 < nt && t >= (I + 1) * nt - (I + 1) * I / 2) ++I;
  const int J = I + t - (I * nt - I * (I - 1) / 2);
  const int i = I * GJ_B + r, j = J * GJ_B + c;
  const bool in = i < N && j < N;
  const int ii = I * GJ_B + c;
  // Y_i^H Y_j, with L^-1 in the block's own place: L^-H Y = P R in its rows, Y^H L^-1 = (P R)^H above it, P on it
  X[r][c] = I == p ? Li[threadIdx.x] : (ii < N ? Y[(long long)r * N + ii] : zero);
  Z[r][c] = J == p ? Li[threadIdx.x] : (j < N ? Y[(long long)r * N + j] : zero);
  double2 v = in && I != p && J != p ? A[(long long)i * N + j] : zero;
  __syncthreads();
  double2 acc = zero;
#pragma unroll
  for (int l = 0; l < GJ_B; ++l) cfmac(acc, X[l][r], Z[l][c]);
  v = I <= p ? cadd(v, acc) : csub(v, acc);
  if (in) A[(long long)i * N + j] = v;
  const int n1 = p + 1;
  if (I == n1) {
    if (j < N) Rn[(long long)r * N + j] = i < N ? v : zero;
  } else if (J == n1) {  // R of the swept columns: -A_i1^H, written by rows (c: row of the tile, r: column of the panel)
    __syncthreads();
    X[r][c] = in ? v : zero;
    __syncthreads();
    if (ii < N) Rn[(long long)r * N + ii] = make_double2(-X[c][r].x, X[c][r].y);
  }
  if (I == p + 2 && J == I)
    g.D[(2 * par + z) * GJ_B * GJ_B + threadIdx.x] = in ? v : make_double2(r == c ? 1.0 : 0.0, 0.0);
}

// Lower triangle from the upper one, tile by tile through shared memory.
__global__ __launch_bounds__(256) void k_gj_mirror(double2* __restrict__ A0, int N, int nt) {
  __shared__ double2 X[GJ_B][GJ_B + 1];
  const int I = blockIdx.x, J = blockIdx.y;
  if (I > J) return;
  double2* A = A0 + (long long)blockIdx.z * N * N;
  const int r = threadIdx.x >> 4, c = threadIdx.x & 15;
  const int i = I * GJ_B + r, j = J * GJ_B + c;
  if (i < N && j < N) X[r][c] = A[(long long)i * N + j];
  __syncthreads();
  const int ti = J * GJ_B + r, tj = I * GJ_B + c;
  if (ti < N && tj < N && ti > tj) A[(long long)ti * N + tj] = cconj(X[c][r]);
}

// Copies the f1 and f2 Toeplitz operators into the workspace that is inverted in place.
__global__ void k_copy2(const double2* __restrict__ src, double2* __restrict__ dst, long long n) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) dst[t] = src[t];
}

// ---------------------------------------------------------------------------
int launch_setup(const SetupArgs& a, cudaStream_t s) {
  const int ne = a.n0 * a.n1 * a.n2;
  const int L = 4 * a.M + 1;
  const int N = (2 * a.M + 1) * (2 * a.M + 1) * (2 * a.M + 1);
  k_interp<<<cdiv(ne, 256), 256, 0, s>>>(a.rho, ne, a.mc, a.fields, a.dchi, a.chi, a.status, a.dfc);
  PC_LAUNCH_CHECK();
  k_mean<<<1, 1024, 0, s>>>(a.chi, ne, a.chi_mean);
  PC_LAUNCH_CHECK();
  long long t1n = 3LL * a.n0 * a.n1 * L;
  k_sfac1<<<cdiv(t1n, 256), 256, 0, s>>>(a.fields, a.n0, a.n1, a.n2, a.M, a.t1);
  PC_LAUNCH_CHECK();
  long long t2n = 3LL * a.n0 * L * L;
  k_sfac2<<<cdiv(t2n, 256), 256, 0, s>>>(a.t1, a.n0, a.n1, a.M, a.t2);
  PC_LAUNCH_CHECK();
  long long sfn = 3LL * L * L * L;
  k_sfac3<<<cdiv(sfn, 256), 256, 0, s>>>(a.t2, a.n0, a.M, 1.0 / (double)ne, a.sfac);
  PC_LAUNCH_CHECK();
  long long NN = (long long)N * N;
  k_toeplitz<<<cdiv(3 * NN, 256), 256, 0, s>>>(a.sfac, a.M, a.V, a.T);
  PC_LAUNCH_CHECK();
  // W1 = T_f1^-1, W2 = T_f2^-1
  k_copy2<<<cdiv(2 * NN, 256), 256, 0, s>>>(a.T + NN, a.W, 2 * NN);
  PC_LAUNCH_CHECK();
  const int nt = cdiv(N, GJ_B);
  GjBufs g;
  g.A = a.W;
  g.R = a.gj;
  g.Y = g.R + 4LL * GJ_B * N;
  g.Li = g.Y + 2LL * GJ_B * N;
  g.D = g.Li + 4LL * GJ_B * GJ_B;
  k_gj_start<<<dim3(nt, 2), 256, 0, s>>>(g, N);
  PC_LAUNCH_CHECK();
  for (int p = 0; p < nt; ++p) {
    k_gj_panel<<<dim3(nt, 2), 256, 0, s>>>(g, N, p & 1);
    PC_LAUNCH_CHECK();
    k_gj_update<<<dim3(1 + nt * (nt + 1) / 2, 2), 256, 0, s>>>(g, N, p, nt);
    PC_LAUNCH_CHECK();
  }
  k_gj_mirror<<<dim3(nt, nt, 2), 256, 0, s>>>(a.W, N, nt);
  PC_LAUNCH_CHECK();
  return PC_OK;
}

// double2 elements of SetupArgs::gj for N plane waves.
long long setup_gj_scratch(int N) { return 6LL * GJ_B * N + 8LL * GJ_B * GJ_B; }

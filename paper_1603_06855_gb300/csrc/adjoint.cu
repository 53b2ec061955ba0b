// Gap objective (Methods, eq. obj; omega form of the Results' note on normalized gaps)
// and the adjoint design sensitivities (Methods, eqs. normalev, sensitivityew, diffOmega,
// diffPhi).  With theta^H Omega theta = 1 and s = Phi^-1 H^H theta,
//   d lambda / d rho_e = chi'_e v_e [ -lambda (rho1 - rho0) sum_c |u_c(x_e)|^2
//                                      - f1'_e |sigma_bulk(x_e)|^2 - f2'_e |sigma_dev(x_e)|^2 ],
// f1'_e, f2'_e the derivatives of the compliance moduli with respect to chi at element e (the
// phase differences under the compliance law, per element under eq. combinematerial's law),
// where u and sigma are the displacement and stress fields synthesised at the element
// centroid from the plane-wave coefficients.  The kernels synthesise the 3 + 6 fields of
// every weighted (k, band) on the voxel grid by separable sums (axis 2, axis 1 into a
// scratch array, then axis 0 inside the per-voxel reduction) and reduce the weighted
// quadratic forms over all (k, band): per chunk of pairs, then over the chunks in FP64.
#include <algorithm>
#include "kernels.h"
#include "launch_rules.h"

// ---------------------------------------------------------------------------
__global__ void k_omega(const double* __restrict__ lam_m, int nk, int nb, int m, double lref,
                        double* __restrict__ omega, double* __restrict__ lam_phys, double* __restrict__ lam_nd) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nk * nb) return;
  int k = t / nb, b = t % nb;
  double l = lam_m[k * m + b];
  if (lam_nd) lam_nd[t] = l;
  if (lam_phys) lam_phys[t] = l * lref;
  if (omega) omega[t] = sqrt(fmax(l * lref, 0.0));
}
int launch_omega(const double* lam_m, int nk, int nb, int m, double lref, double* omega, double* lam_nd,
                 cudaStream_t s) {
  k_omega<<<cdiv((long long)nk * nb, 256), 256, 0, s>>>(lam_m, nk, nb, m, lref, omega, nullptr, lam_nd);
  PC_LAUNCH_CHECK();
  return PC_OK;
}

// ---------------------------------------------------------------------------
// Gap, weights dG/dlambda (physical) and the compacted list of weighted (k, band).
__global__ void k_gap(GapArgs a) {
  __shared__ double sv[256];
  __shared__ int si[256];
  __shared__ int ka_s, kb_s;
  const int nk = a.nk, nb = a.nb;
  for (int t = threadIdx.x; t < nk * nb; t += blockDim.x) a.weights[t] = 0.0;
  __syncthreads();
  if (a.mode == PC_GRAD_ALLBANDS) {
    double s = 0.0;
    for (int t = threadIdx.x; t < nk * nb; t += blockDim.x) {
      a.weights[t] = a.w_user[t];
      s += a.w_user[t] * a.lam[t] * a.lref;
    }
    sv[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
      if ((int)threadIdx.x < w) sv[threadIdx.x] += sv[threadIdx.x + w];
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      *a.gap_out = sv[0];
      int c = 0;
      for (int t = 0; t < nk * nb; ++t)
        if (a.weights[t] != 0.0) a.pairs[c++] = t;
      *a.npairs = c;
    }
    return;
  }
  const int lo = a.n_lower - 1, hi = a.n_lower;
  if (a.mode == PC_GAP_KS_INTERNAL) {
    // Smooth surrogate: with x = omega / omega_ref = sqrt(lam_nd), a = (1/beta) log sum_k
    // exp(beta x_{k,lo}) and b = -(1/beta) log sum_k exp(-beta x_{k,hi}), G = 2 (b - a) / (b + a).
    __shared__ double xm_s, ym_s, sa_s, sb_s;
    const double beta = a.ks_beta;
    double mx = -1e300, my = 1e300;
    for (int k = threadIdx.x; k < nk; k += blockDim.x) {
      mx = fmax(mx, sqrt(fmax(a.lam[k * nb + lo], 0.0)));
      my = fmin(my, sqrt(fmax(a.lam[k * nb + hi], 0.0)));
    }
    sv[threadIdx.x] = mx;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
      if ((int)threadIdx.x < w) sv[threadIdx.x] = fmax(sv[threadIdx.x], sv[threadIdx.x + w]);
      __syncthreads();
    }
    if (threadIdx.x == 0) xm_s = sv[0];
    __syncthreads();
    sv[threadIdx.x] = my;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
      if ((int)threadIdx.x < w) sv[threadIdx.x] = fmin(sv[threadIdx.x], sv[threadIdx.x + w]);
      __syncthreads();
    }
    if (threadIdx.x == 0) ym_s = sv[0];
    __syncthreads();
    const double xm = xm_s, ym = ym_s;
    double pa = 0.0, pb = 0.0;
    for (int k = threadIdx.x; k < nk; k += blockDim.x) {
      pa += exp(beta * (sqrt(fmax(a.lam[k * nb + lo], 0.0)) - xm));
      pb += exp(-beta * (sqrt(fmax(a.lam[k * nb + hi], 0.0)) - ym));
    }
    sv[threadIdx.x] = pa;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
      if ((int)threadIdx.x < w) sv[threadIdx.x] += sv[threadIdx.x + w];
      __syncthreads();
    }
    if (threadIdx.x == 0) sa_s = sv[0];
    __syncthreads();
    sv[threadIdx.x] = pb;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
      if ((int)threadIdx.x < w) sv[threadIdx.x] += sv[threadIdx.x + w];
      __syncthreads();
    }
    if (threadIdx.x == 0) sb_s = sv[0];
    __syncthreads();
    const double A_ = xm + log(sa_s) / beta, B_ = ym - log(sb_s) / beta;
    const double dGa = -4.0 * B_ / ((A_ + B_) * (A_ + B_)), dGb = 4.0 * A_ / ((A_ + B_) * (A_ + B_));
    if (threadIdx.x == 0) *a.gap_out = 2.0 * (B_ - A_) / (B_ + A_);
    // weights dG/dlambda_phys: p_k dGa / (2 x lref) on band lo, q_k dGb / (2 y lref) on band hi,
    // each shared by the bands of its cluster at that k (one thread per k: no write conflicts)
    for (int k = threadIdx.x; k < nk; k += blockDim.x) {
      for (int side = 0; side < 2; ++side) {
        const int band = side == 0 ? lo : hi;
        const double xv = sqrt(fmax(a.lam[k * nb + band], 0.0));
        if (xv <= 0.0) continue;
        const double pw = side == 0 ? exp(beta * (xv - xm)) / sa_s : exp(-beta * (xv - ym)) / sb_s;
        const double wl = (side == 0 ? dGa : dGb) * pw / (2.0 * xv * a.lref);
        const double ref = a.lam[k * nb + band];
        int members = 0;
        for (int b = 0; b < nb; ++b) members += (fabs(a.lam[k * nb + b] - ref) <= a.rel_tol * fabs(ref)) ? 1 : 0;
        for (int b = 0; b < nb; ++b)
          if (fabs(a.lam[k * nb + b] - ref) <= a.rel_tol * fabs(ref)) a.weights[k * nb + b] += wl / members;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int c = 0;
      for (int t = 0; t < nk * nb; ++t)
        if (a.weights[t] != 0.0) a.pairs[c++] = t;
      *a.npairs = c;
    }
    return;
  }
  // argmax_k lam[k][lo], lowest k among ties
  double bv = -1e300;
  int bi = 0x7fffffff;
  for (int k = threadIdx.x; k < nk; k += blockDim.x) {
    double v = a.lam[k * nb + lo];
    if (v > bv || (v == bv && k < bi)) { bv = v; bi = k; }
  }
  sv[threadIdx.x] = bv; si[threadIdx.x] = bi;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      double v2 = sv[threadIdx.x + w]; int i2 = si[threadIdx.x + w];
      if (v2 > sv[threadIdx.x] || (v2 == sv[threadIdx.x] && i2 < si[threadIdx.x])) { sv[threadIdx.x] = v2; si[threadIdx.x] = i2; }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) ka_s = si[0];
  __syncthreads();
  // argmin_k lam[k][hi], lowest k among ties
  bv = 1e300; bi = 0x7fffffff;
  for (int k = threadIdx.x; k < nk; k += blockDim.x) {
    double v = a.lam[k * nb + hi];
    if (v < bv || (v == bv && k < bi)) { bv = v; bi = k; }
  }
  sv[threadIdx.x] = bv; si[threadIdx.x] = bi;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      double v2 = sv[threadIdx.x + w]; int i2 = si[threadIdx.x + w];
      if (v2 < sv[threadIdx.x] || (v2 == sv[threadIdx.x] && i2 < si[threadIdx.x])) { sv[threadIdx.x] = v2; si[threadIdx.x] = i2; }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) kb_s = si[0];
  __syncthreads();
  if (threadIdx.x != 0) return;
  int ka = ka_s, kb = kb_s;
  double la = a.lam[ka * nb + lo] * a.lref, lb = a.lam[kb * nb + hi] * a.lref;
  double G, wa, wb;
  if (a.mode == PC_GAP_OMEGA) {
    double A_ = sqrt(fmax(la, 0.0)), B_ = sqrt(fmax(lb, 0.0));
    G = 2.0 * (B_ - A_) / (B_ + A_);
    wa = A_ > 0.0 ? -2.0 * B_ / (A_ * (A_ + B_) * (A_ + B_)) : 0.0;
    wb = B_ > 0.0 ? 2.0 * A_ / (B_ * (A_ + B_) * (A_ + B_)) : 0.0;
  } else {
    G = 2.0 * (lb - la) / (lb + la);
    wa = -4.0 * lb / ((la + lb) * (la + lb));
    wb = 4.0 * la / ((la + lb) * (la + lb));
  }
  *a.gap_out = G;
  int c = 0;
  for (int side = 0; side < 2; ++side) {
    int k = side == 0 ? ka : kb;
    int band = side == 0 ? lo : hi;
    double wt = side == 0 ? wa : wb;
    double ref = a.lam[k * nb + band];
    int members = 0;
    for (int b = 0; b < nb; ++b) members += (fabs(a.lam[k * nb + b] - ref) <= a.rel_tol * fabs(ref)) ? 1 : 0;
    for (int b = 0; b < nb; ++b)
      if (fabs(a.lam[k * nb + b] - ref) <= a.rel_tol * fabs(ref)) a.weights[k * nb + b] += wt / members;
  }
  for (int t = 0; t < nk * nb; ++t)
    if (a.weights[t] != 0.0) a.pairs[c++] = t;
  *a.npairs = c;
}
int launch_gap(const GapArgs& a, cudaStream_t s) {
  k_gap<<<1, 256, 0, s>>>(a);
  PC_LAUNCH_CHECK();
  return PC_OK;
}

// ---------------------------------------------------------------------------
// Phases of the synthesis.  Voxel centroids sit at (2 i + 1) / (2 n), so that voxels i and n - 1 - i have
// conjugate phases: with s_g = x_g + x_-g and d_g = x_g - x_-g,
//   sum_g x_g e^{i pi g (2i+1)/n} = x_0 + sum_{g>0} s_g cos + i sum_{g>0} d_g sin,
// and its conjugate phases give the mirrored voxel from the same two sums: 4 M real multiply-adds for two
// voxels instead of 8 (2M + 1).  ph: (cos, sin) of pi g (2i+1)/n, [axis][g - 1][i].
template <typename R>
__global__ void k_adj_phases(int M, int n0, int n1, int n2, typename cplx_t<R>::type* __restrict__ ph) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int n = n0 + n1 + n2;
  if (t >= M * n) return;
  const int first[4] = {0, M * n0, M * (n0 + n1), M * n};
  const int ax = t >= first[2] ? 2 : (t >= first[1] ? 1 : 0);
  const int len = ax == 0 ? n0 : (ax == 1 ? n1 : n2), r = t - first[ax];
  ph[t] = from_d2<R>(phase_pi_over((long long)(r / len + 1) * (2 * (r % len) + 1), len));
}
int launch_adj_phases(int M, const int n[3], bool fp32, void* ph, cudaStream_t s) {
  const int c = cdiv((long long)M * (n[0] + n[1] + n[2]), 128);
  if (fp32) k_adj_phases<float><<<c, 128, 0, s>>>(M, n[0], n[1], n[2], (float2*)ph);
  else k_adj_phases<double><<<c, 128, 0, s>>>(M, n[0], n[1], n[2], (double2*)ph);
  PC_LAUNCH_CHECK();
  return PC_OK;
}
// The two sums from (x_0, s, d) and the phases: z the voxel, zm its mirror image.
template <typename R, int M, typename C2 = typename cplx_t<R>::type>
__device__ __forceinline__ void mirror_pair(C2 x0, const C2 (&s)[M], const C2 (&d)[M], const C2 (&ph)[M], C2& z, C2& zm) {
  C2 c = x0, t = mk<R>(0, 0);
#pragma unroll
  for (int g = 0; g < M; ++g) {
    c.x += s[g].x * ph[g].x; c.y += s[g].y * ph[g].x;
    t.x += d[g].x * ph[g].y; t.y += d[g].y * ph[g].y;
  }
  z = mk<R>(c.x - t.y, c.y + t.x);
  zm = mk<R>(c.x + t.y, c.y - t.x);
}

// Axis-2 and axis-1 synthesis of field f of pair p:
//   t2[p][f][g1][j][l] = sum_{g2,g3} c[g1][g2][g3] e^{i pi G2 (2j+1)/n1} e^{i pi G3 (2l+1)/n2}
// f < 3: displacement component f of theta; f >= 3: stress coordinate f-3.  R is the
// arithmetic of the synthesis (FP64 for the FP64 form, FP32 for the mixed form).
// One CTA per field and pair.  Axis 1: a thread keeps the column (g1, ., l) in registers and runs over its
// share of the mirrored pairs of j, so that a value costs one broadcast load and 2 M multiply-adds.
// 48^3, M = 3, 720 pairs (836 MB of t2, 0.13 ms): 0.68 ms with
// a full sum per value and FP64 sincospi per CTA, 0.14 ms.
template <typename R, int M>
__global__ __launch_bounds__(256) void k_adj_synth12(AdjointArgs a, int jsplit) {
  typedef typename cplx_t<R>::type C2;
  constexpr int M2 = 2 * M + 1, N = M2 * M2 * M2;
  extern __shared__ __align__(16) unsigned char smem[];
  const int p = blockIdx.x, f = blockIdx.y;
  if (p >= *a.npairs) return;
  const int n1 = a.n1, n2 = a.n2;
  C2* c = (C2*)smem;                 // N
  C2* t1 = c + N;                    // M2*M2*n2
  C2* ph3 = t1 + M2 * M2 * n2;       // M*n2
  C2* ph2 = ph3 + M * n2;            // M*n1
  const int pr = a.pairs[p];
  const int k = pr / a.nb, b = pr % a.nb;
  const long long vec = (long long)k * a.m + b;
  const long long nvec = (long long)a.nk * a.m;
  const double2* src = (f < 3) ? a.theta + (vec * 3 + f) * N : a.sig + ((long long)(f - 3) * nvec + vec) * N;
  const C2* tab = (const C2*)a.phases;
  for (int q = threadIdx.x; q < N; q += blockDim.x) c[q] = from_d2<R>(src[q]);
  for (int t = threadIdx.x; t < M * n2; t += blockDim.x) ph3[t] = tab[M * (a.n0 + n1) + t];
  for (int t = threadIdx.x; t < M * n1; t += blockDim.x) ph2[t] = tab[M * a.n0 + t];
  __syncthreads();
  const int h2 = (n2 + 1) / 2, h1 = (n1 + 1) / 2;
  C2 s[M], d[M], ph[M], z, zm;
  for (int t = threadIdx.x; t < M2 * M2 * h2; t += blockDim.x) {
    const int g12 = t / h2, l = t % h2;
    const C2* x = c + g12 * M2 + M;
#pragma unroll
    for (int g = 0; g < M; ++g) {
      s[g] = cadd(x[g + 1], x[-g - 1]);
      d[g] = mk<R>(x[g + 1].x - x[-g - 1].x, x[g + 1].y - x[-g - 1].y);
      ph[g] = ph3[g * n2 + l];
    }
    mirror_pair<R, M>(x[0], s, d, ph, z, zm);
    t1[g12 * n2 + l] = z;
    t1[g12 * n2 + n2 - 1 - l] = zm;
  }
  __syncthreads();
  C2* out = (C2*)a.t2 + ((long long)p * 9 + f) * M2 * n1 * n2;
  for (int t = threadIdx.x; t < jsplit * M2 * n2; t += blockDim.x) {
    const int l = t % n2, g1 = (t / n2) % M2, jq = t / (n2 * M2);
    const C2* x = t1 + (g1 * M2 + M) * n2 + l;
#pragma unroll
    for (int g = 0; g < M; ++g) {
      const C2 u = x[(g + 1) * n2], v = x[-(g + 1) * n2];
      s[g] = cadd(u, v);
      d[g] = mk<R>(u.x - v.x, u.y - v.y);
    }
    const C2 x0 = x[0];
    C2* o = out + (long long)g1 * n1 * n2 + l;
    for (int j = jq; j < h1; j += jsplit) {
#pragma unroll
      for (int g = 0; g < M; ++g) ph[g] = ph2[g * n1 + j];
      mirror_pair<R, M>(x0, s, d, ph, z, zm);
      o[j * n2] = z;
      o[(n1 - 1 - j) * n2] = zm;
    }
  }
}

// Axis-0 synthesis fused with the weighted reduction over (k, band).  The pairs are cut into
// chunks along the grid's z; each thread synthesises V mirrored pairs of voxels along axis 0 at one (j, l), so
// that every loaded axis-1/2 coefficient feeds 2 V voxels, and sums its chunk's three
// weighted quadratic forms in R (FP32 in the mixed form: at most 128 pairs, adj_chunks in launch_rules.h).  The
// chunk sums go to part[chunk][3][ne]; k_adj_finish adds them in FP64 in chunk order.
// A warp takes 32 columns (j, l) of one group of V pairs; the warps of a CTA take the groups of the same columns
// and share their coefficients through a ring of kAdjStages pairs in shared memory, filled by asynchronous
// copies two pairs ahead, so that each comes from L2 once.
// Bound: instruction issue (48^3, M = 3, 720 pairs: 0.25 ms; 836 MB of t2 at the copy rate 0.13 ms).  A full sum
// per voxel, FP64 sincospi per thread and loads from L2 where they are used took 1.77 ms, the mirrored sums with
// tabulated phases 0.83 ms, the ring 0.47 ms.
constexpr int kAdjReduceWarps = 8;
constexpr int kAdjStages = 3;

template <typename R, int M, int V>
__global__ __launch_bounds__(32 * kAdjReduceWarps) void k_adj_reduce(AdjointArgs a, int chunk) {
  typedef typename cplx_t<R>::type C2;
  constexpr int M2 = 2 * M + 1, ROWS = 9 * M2;
  extern __shared__ __align__(16) unsigned char adj_ring[];
  C2* ring = (C2*)adj_ring;  // [kAdjStages][ROWS][32]
  const int np = *a.npairs;
  if ((int)blockIdx.z * chunk >= np) return;  // k_adj_finish leaves this chunk out
  const int n0 = a.n0, h0 = (n0 + 1) / 2, lane = threadIdx.x;
  const long long jl = (long long)a.n1 * a.n2;
  const long long v = (long long)blockIdx.x * 32 + lane, vc = v < jl ? v : jl - 1;
  const int ig = blockIdx.y * blockDim.y + threadIdx.y;
  const C2* tab = (const C2*)a.phases;
  C2 ph[V][M];  // compile-time sizes and fully unrolled loops keep these in registers
#pragma unroll
  for (int s = 0; s < V; ++s)
#pragma unroll
    for (int g = 0; g < M; ++g) ph[s][g] = tab[g * n0 + min(ig * V + s, h0 - 1)];
  const int p0 = blockIdx.z * chunk, p1 = min(np, p0 + chunk);
  const C2* t2 = (const C2*)a.t2 + vc;
  auto fill = [&](int p) {  // one group per call, empty past the end, so that the wait counts are constant
    if (p < p1) {
      C2* to = ring + (p - p0) % kAdjStages * ROWS * 32 + lane;
      const C2* from = t2 + (long long)p * ROWS * jl;
      for (int r = threadIdx.y; r < ROWS; r += blockDim.y)
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(to + r * 32)),
                     "l"(from + r * jl), "n"((int)sizeof(C2))
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // the compliance part's factors d f1/d chi, d f2/d chi belong to the element: three weighted sums, of
  // the voxels and of their mirror images
  R acc_m[2][V], acc_1[2][V], acc_2[2][V];
#pragma unroll
  for (int s = 0; s < V; ++s)
#pragma unroll
    for (int h = 0; h < 2; ++h) acc_m[h][s] = acc_1[h][s] = acc_2[h][s] = (R)0;
  for (int i = 0; i < kAdjStages - 1; ++i) fill(p0 + i);
  for (int p = p0; p < p1; ++p) {
    const int pr = a.pairs[p];
    const double wd = a.weights[pr];
    const R w = (R)(wd * a.w_scale), wl = (R)(wd * a.lam[pr] * a.lref);
    asm volatile("cp.async.wait_group %0;" ::"n"(kAdjStages - 2) : "memory");
    __syncthreads();  // pair p is there, and every warp is done with pair p - 1, whose slot is filled now
    fill(p + kAdjStages - 1);
    const C2* base = ring + (p - p0) % kAdjStages * ROWS * 32 + lane;
    R q[2][V];
#pragma unroll
    for (int f = 0; f < 9; ++f) {
      if (f == 0 || f == 3 || f == 4) {
#pragma unroll
        for (int s = 0; s < V; ++s) q[0][s] = q[1][s] = (R)0;
      }
      C2 x[M2], sg[M], d[M];
#pragma unroll
      for (int g = 0; g < M2; ++g) x[g] = base[(f * M2 + g) * 32];
#pragma unroll
      for (int g = 0; g < M; ++g) {
        sg[g] = cadd(x[M + 1 + g], x[M - 1 - g]);
        d[g] = mk<R>(x[M + 1 + g].x - x[M - 1 - g].x, x[M + 1 + g].y - x[M - 1 - g].y);
      }
#pragma unroll
      for (int s = 0; s < V; ++s) {
        C2 z, zm;
        mirror_pair<R, M>(x[M], sg, d, ph[s], z, zm);
        q[0][s] += z.x * z.x + z.y * z.y;
        q[1][s] += zm.x * zm.x + zm.y * zm.y;
      }
#pragma unroll
      for (int s = 0; s < V; ++s)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (f == 2) acc_m[h][s] += wl * q[h][s];
          if (f == 3) acc_1[h][s] += w * q[h][s];
          if (f == 8) acc_2[h][s] += w * q[h][s];
        }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if (v >= jl) return;
  const long long ne = n0 * jl;
  R* part = (R*)a.part + (long long)blockIdx.z * 3 * ne + v;
#pragma unroll
  for (int s = 0; s < V; ++s) {
    const int i = ig * V + s;
    if (i >= h0) break;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const long long e = (h ? n0 - 1 - i : i) * jl;
      part[e] = acc_m[h][s];
      part[ne + e] = acc_1[h][s];
      part[2 * ne + e] = acc_2[h][s];
    }
  }
}

// The chunk sums added in FP64 and combined with the per-element factors.
template <typename R>
__global__ void k_adj_finish(AdjointArgs a, int chunk) {
  const long long ne = (long long)a.n0 * a.n1 * a.n2;
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= ne) return;
  const R* part = (const R*)a.part;
  const int nchunks = (*a.npairs + chunk - 1) / chunk;
  double acc_m = 0.0, acc_1 = 0.0, acc_2 = 0.0;
  for (int c = 0; c < nchunks; ++c) {
    const R* pc = part + (long long)c * 3 * ne;
    acc_m += (double)pc[e];
    acc_1 += (double)pc[ne + e];
    acc_2 += (double)pc[2 * ne + e];
  }
  const double acc = -a.d_rho * acc_m - a.two_pi_V_sq * (a.w_inv * (a.dfc[e] * acc_1 + a.dfc[ne + e] * acc_2));
  a.grad[e] = acc * a.inv_sO * a.ve * a.dchi[e];
}

size_t adjoint_staging_bytes(int M, int n1, int n2, bool fp32) {
  const size_t M2 = 2 * (size_t)M + 1;
  const size_t elems = M2 * M2 * M2 + M2 * M2 * (size_t)n2 + M2 * (size_t)n2 + M2 * (size_t)n1;
  return elems * (fp32 ? sizeof(float2) : sizeof(double2));
}

// Mirrored pairs per thread of the reduction: 4 in FP32 (2 at M = 5), 1 in FP64 (registers).
template <typename R>
constexpr int adj_pairs(int M) { return sizeof(R) == sizeof(float) ? (M <= 4 ? 4 : 2) : 1; }

template <typename R, int M>
static int launch_adjoint_m(const AdjointArgs& a, cudaStream_t s) {
  constexpr int M2 = 2 * M + 1, V = adj_pairs<R>(M);
  const size_t sm = adjoint_staging_bytes(a.M, a.n1, a.n2, sizeof(R) == sizeof(float));
  // Set once per instantiation; a function-local static is initialised exactly once even when
  // k groups on several host threads arrive together.
  static const cudaError_t attr =
      cudaFuncSetAttribute(k_adj_synth12<R, M>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kAdjointStagingMax);
  (void)attr;
  if (sm > kAdjointStagingMax) return PC_EINVAL;
  dim3 g1(a.max_pairs, 9);
  const int jsplit = std::max(1, std::min((a.n1 + 1) / 2, (int)cdiv(768, M2 * a.n2)));
  k_adj_synth12<R, M><<<g1, 256, sm, s>>>(a, jsplit);
  PC_LAUNCH_CHECK();
  const int h0 = (a.n0 + 1) / 2;
  const int nig = (int)cdiv(h0, V), wy = std::min(nig, kAdjReduceWarps);
  const dim3 block(32, wy);
  dim3 grid((unsigned)cdiv((long long)a.n1 * a.n2, 32), (unsigned)cdiv(nig, wy));
  // as many pair chunks as are resident at once, or a multiple, so that no last wave is nearly empty; the chunks
  // cover max_pairs, and the ones past the device's pair count are left out
  constexpr size_t ring = sizeof(typename cplx_t<R>::type) * kAdjStages * 9 * M2 * 32;
  static const cudaError_t rattr =
      cudaFuncSetAttribute(k_adj_reduce<R, M, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ring);
  (void)rattr;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_adj_reduce<R, M, V>, 32 * wy, ring) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  int nchunks = (int)std::min<long long>(kAdjChunksMax, std::max<long long>(1, (long long)per_sm * device_sms() / (grid.x * grid.y)));
  nchunks = std::max(1, std::min(nchunks, a.max_pairs));
  // (the room for kAdjChunksMax FP64 sums a voxel holds twice as many in FP32)
  if (sizeof(R) == sizeof(float)) nchunks = adj_chunks(a.max_pairs, nchunks, 2 * kAdjChunksMax);
  const int chunk = (int)cdiv(a.max_pairs, nchunks);
  nchunks = (int)cdiv(a.max_pairs, chunk);
  grid.z = nchunks;
  k_adj_reduce<R, M, V><<<grid, block, ring, s>>>(a, chunk);
  PC_LAUNCH_CHECK();
  const long long ne = (long long)a.n0 * a.n1 * a.n2;
  k_adj_finish<R><<<(unsigned)cdiv(ne, 256), 256, 0, s>>>(a, chunk);
  PC_LAUNCH_CHECK();
  return PC_OK;
}
template <typename R>
static int launch_adjoint_t(const AdjointArgs& a, cudaStream_t s) {
  switch (a.M) {
    case 1: return launch_adjoint_m<R, 1>(a, s);
    case 2: return launch_adjoint_m<R, 2>(a, s);
    case 3: return launch_adjoint_m<R, 3>(a, s);
    case 4: return launch_adjoint_m<R, 4>(a, s);
    case 5: return launch_adjoint_m<R, 5>(a, s);
    default: return PC_EINVAL;
  }
}

int launch_adjoint(const AdjointArgs& a, bool fp32, cudaStream_t s) {
  return fp32 ? launch_adjoint_t<float>(a, s) : launch_adjoint_t<double>(a, s);
}

// Per plane wave arithmetic shared by the operator and preconditioner kernels: wavevectors, the strain
// coordinates of the operator and their transpose, the reference medium's resolvent.
#pragma once
#include "kernels.h"

#define RS2 0.70710678118654752440
#define RS3 0.57735026918962576451
#define RS6 0.40824829046386301637

__device__ __forceinline__ void kvec(const Geom& g, const double* Q, int k, int q, double K[3]) {
  int M2 = 2 * g.M + 1;
  double a0 = Q[3 * k + 0] + (double)(q / (M2 * M2) - g.M);
  double a1 = Q[3 * k + 1] + (double)((q / M2) % M2 - g.M);
  double a2 = Q[3 * k + 2] + (double)(q % M2 - g.M);
  K[0] = g.T[0] * a0 + g.T[1] * a1 + g.T[2] * a2;
  K[1] = g.T[3] * a0 + g.T[4] * a1 + g.T[5] * a2;
  K[2] = g.T[6] * a0 + g.T[7] * a1 + g.T[8] * a2;
}

// The FP32 components of K at (k, q): from the table when there is one (FP32 data only).
template <typename R>
__device__ __forceinline__ void kvec_r(const Geom& g, const double* Q, const float4* Kf, int k, int q, R& k0, R& k1,
                                       R& k2) {
  if (Kf) {
    const float4 kk = Kf[(long long)k * g.N + q];
    k0 = (R)kk.x; k1 = (R)kk.y; k2 = (R)kk.z;
  } else {
    double K[3];
    kvec(g, Q, k, q, K);
    k0 = (R)K[0]; k1 = (R)K[1]; k2 = (R)K[2];
  }
}

// The six strain coordinates of the displacement coefficients u of plane wave K.
template <typename R, typename C2 = typename cplx_t<R>::type>
__device__ __forceinline__ void strain6(R k0, R k1, R k2, C2 u0, C2 u1, C2 u2, C2 e[6]) {
  e[0] = mk<R>((k0 * u0.x + k1 * u1.x + k2 * u2.x) * (R)RS3, (k0 * u0.y + k1 * u1.y + k2 * u2.y) * (R)RS3);
  e[1] = mk<R>((k0 * u0.x - k1 * u1.x) * (R)RS2, (k0 * u0.y - k1 * u1.y) * (R)RS2);
  e[2] = mk<R>((k0 * u0.x + k1 * u1.x - 2 * k2 * u2.x) * (R)RS6, (k0 * u0.y + k1 * u1.y - 2 * k2 * u2.y) * (R)RS6);
  e[3] = mk<R>((k1 * u2.x + k2 * u1.x) * (R)RS2, (k1 * u2.y + k2 * u1.y) * (R)RS2);
  e[4] = mk<R>((k0 * u2.x + k2 * u0.x) * (R)RS2, (k0 * u2.y + k2 * u0.y) * (R)RS2);
  e[5] = mk<R>((k0 * u1.x + k1 * u0.x) * (R)RS2, (k0 * u1.y + k1 * u0.y) * (R)RS2);
}
// Its transpose: the force o of the six stress coordinates sg (stride st), bulk scaled by c0 and deviatoric by c1.
template <typename R, typename C2 = typename cplx_t<R>::type>
__device__ __forceinline__ void strain6_t(R k0, R k1, R k2, const C2* __restrict__ sg, long long st, R c0, R c1, C2 o[3]) {
  const C2 s0 = cscale(sg[0], c0 * (R)RS3);
  const C2 s1 = cscale(sg[st], c1 * (R)RS2), s2 = cscale(sg[2 * st], c1 * (R)RS6);
  const C2 s3 = cscale(sg[3 * st], c1 * (R)RS2), s4 = cscale(sg[4 * st], c1 * (R)RS2), s5 = cscale(sg[5 * st], c1 * (R)RS2);
  // component 1: B_0 = K1/sqrt3, B_1 = K1/sqrt2, B_2 = K1/sqrt6, B_4 = K3/sqrt2, B_5 = K2/sqrt2
  o[0] = mk<R>(k0 * (s0.x + s1.x + s2.x) + k2 * s4.x + k1 * s5.x, k0 * (s0.y + s1.y + s2.y) + k2 * s4.y + k1 * s5.y);
  // component 2: B_0 = K2/sqrt3, B_1 = -K2/sqrt2, B_2 = K2/sqrt6, B_3 = K3/sqrt2, B_5 = K1/sqrt2
  o[1] = mk<R>(k1 * (s0.x - s1.x + s2.x) + k2 * s3.x + k0 * s5.x, k1 * (s0.y - s1.y + s2.y) + k2 * s3.y + k0 * s5.y);
  // component 3: B_0 = K3/sqrt3, B_2 = -2 K3/sqrt6, B_3 = K2/sqrt2, B_4 = K1/sqrt2
  o[2] = mk<R>(k2 * (s0.x - 2 * s2.x) + k1 * s3.x + k0 * s4.x, k2 * (s0.y - 2 * s2.y) + k1 * s3.y + k0 * s4.y);
}

// The preconditioner of the block iteration.  A = B^T W B, and the compliance operators T with T W = 1
// are at hand (the set-up inverts them), so
//     P = R0 [ B^T W0 T W0 B + s ] R0,   R0 = (B^T W0 B + s)^-1,
// with the bulk and shear moduli W0 of a homogeneous reference medium and the shift s: B0 = R0 B^T W0 is
// (up to s) a left inverse of B, and B0 T B0^T inverts A but for the part of the stress that the reference
// medium cannot tell from an incompatible strain.  For a homogeneous cell P = R0, which is what the
// iteration used alone before; on strong contrasts R0 leaves the condition of the contrast, P about its
// square root: the block iterations fall 1.5 to 3 times (level sets, FCC N = 729: 113 -> 54-82; spheres,
// N = 343: 98-221 -> 37-69; random fields 14-32 -> 11-17) for one more product of two thirds of the operator's.
// R0 is diagonal in the plane waves: (a I + b K K^T)^-1 = (I - b/(a + b|K|^2) K K^T) / a with
// a = mu |K|^2 + s, b = lambda + mu.
template <typename R>
struct PrecTerm {
  R w1, w2, s;  // 3 kappa and 2 mu of the reference medium, shift at this k-point (nondimensional)
  // ref: PrecRefVals; lam: the k-point's Ritz values, nb wanted
  __device__ __forceinline__ PrecTerm(const double* __restrict__ ref, const R* __restrict__ lam, int nb) {
    w1 = (R)ref[0];
    w2 = (R)ref[1];
    R sig = 0;
    for (int j = 0; j < nb; ++j) sig = fmax(sig, lam[j]);
    s = fmax(sig, (R)1e-6) * (R)ref[2];
  }
  template <typename C2>
  __device__ __forceinline__ void solve(R k0, R k1, R k2, C2 u[3]) const {  // u <- R0 u
    const R mu = (R)0.5 * w2, b = (w1 - w2) * (R)(1.0 / 3.0) + mu;
    const R kk = k0 * k0 + k1 * k1 + k2 * k2;
    const R a = mu * kk + s, ia = (R)1 / a, f = b / (a + b * kk);
    const R kx = f * (k0 * u[0].x + k1 * u[1].x + k2 * u[2].x), ky = f * (k0 * u[0].y + k1 * u[1].y + k2 * u[2].y);
    u[0] = mk<R>((u[0].x - k0 * kx) * ia, (u[0].y - k0 * ky) * ia);
    u[1] = mk<R>((u[1].x - k1 * kx) * ia, (u[1].y - k1 * ky) * ia);
    u[2] = mk<R>((u[2].x - k2 * kx) * ia, (u[2].y - k2 * ky) * ia);
  }
};
// u = Y = R0 (A x - l Omega x) at wave q of vector vec (k-point k), stored to Wv, and its strain coordinates e.
template <typename R, typename C2 = typename cplx_t<R>::type>
__device__ __forceinline__ void prec_residual(const PrecTerm<R>& pt, const C2* __restrict__ AX, const C2* __restrict__ OX,
                                              C2* __restrict__ Wv, R l, int vec, const Geom& g, const double* Q,
                                              const float4* Kf, int k, int q, C2 u[3], C2 e[6]) {
  const int N = g.N;
  const long long o = (long long)vec * 3 * N + q;
  R k0, k1, k2;
  kvec_r<R>(g, Q, Kf, k, q, k0, k1, k2);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const C2 av = AX[o + c * N], ov = OX[o + c * N];
    u[c] = mk<R>(av.x - l * ov.x, av.y - l * ov.y);
  }
  pt.solve(k0, k1, k2, u);
#pragma unroll
  for (int c = 0; c < 3; ++c) Wv[o + c * N] = u[c];
  strain6<R>(k0, k1, k2, u[0], u[1], u[2], e);
}

// Design parametrisation (Methods, "Topology optimization formulation", the passage after eq.
// sensitivityew; Results, "Topology optimized structures"): element densities as a closed-form
// function of a reduced design field, and the chain rule back.
//
//   x (free variables) --[SC octant mirror, optional]--> phi (design nodes, every `spacing`
//   elements) --[linear-weight average within the radius]--> mu (elements)
//   --[Heaviside projection]--> rho_e = 1 - exp(-beta mu_e) + mu_e exp(-beta)
//
// Design node a of a spacing-2 grid sits at the centre of the 2 x 2 x 2 element block a,
// fractional position (2a + 1) / n per axis; with spacing 1 the nodes are the element centroids.
// Element e averages the nodes within the radius r with weights w = r - |x_a - x_e| (Cartesian,
// nearest periodic image).  The weight of a node depends only on its offset d (in nodes) from the
// element's block and on the element's position p inside its block (its parity class), so one
// table of (p, d, w) serves every element (forward: gather over the nodes of the element's class)
// and every node (backward: gather over the elements e = spacing (a - d) + p of each class).
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <utility>
#include <vector>
#include "kernels.h"

struct DesignEntry {
  int d0, d1, d2;  // node offset from the element's block
  double w;        // weight / total weight of the class
};

struct pc_design {
  int n[3], nd[3], spacing, octant;
  long long ne, nnodes, nvars;
  int nclass;
  // one device allocation
  double* exp2t = nullptr;       // 2^(j / 64), j < 64
  DesignEntry* table = nullptr;  // entries of class 0, then class 1, ...
  int* class_start = nullptr;    // nclass + 1 offsets into table
  double* dmu = nullptr;         // ne, d rho / d mu of the last projection
  double* gmu = nullptr;         // ne, dG/dmu (large maps); the members below say whose (gmu_claim)
  std::mutex gmu_lock;
  cudaEvent_t gmu_read = nullptr;       // after the last launch that reads gmu
  unsigned long long gmu_stream = 0;    // and the identity of its stream
  bool gmu_used = false;
};

namespace {

__device__ __forceinline__ int wrap(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// fmin(fmax(v, 0), 1), NaN to 0, on the integer units (the FP64 unit is the bound here).
__device__ __forceinline__ double clamp01(double v) {
  const long long b = __double_as_longlong(v);
  if (b < 0 || b > 0x7ff0000000000000LL) return 0.0;
  return b > 0x3ff0000000000000LL ? 1.0 : v;
}

// exp(x) for -690 < x <= 0 by table and polynomial (Tang, ACM Trans. Math. Softw. 15, 1989):
// x = (64 k + j) ln2 / 64 + r, |r| <= ln2 / 128, exp(x) = 2^k 2^(j/64) (1 + r + r^2/2 + ... + r^5/120).
// The remainder r^6/720 is below 4e-17.  10 FP64 instructions.
__device__ __forceinline__ double exp_tab(double x, const double* __restrict__ tab) {
  constexpr double ln2_hi = 6.93147180369123816490e-01;  // ln 2 to 33 bits, and the rest (the split of fdlibm)
  constexpr double ln2_lo = 1.90821492927058770002e-10;
  constexpr double shift = 6755399441055744.0;  // 1.5 2^52: rounds to an integer in the low word
  const double t = fma(x, 64.0 / 0.69314718055994530942, shift);
  const int n = __double2loint(t);
  const double nd = t - shift;
  double r = fma(nd, -ln2_hi / 64.0, x);
  r = fma(nd, -ln2_lo / 64.0, r);
  double p = fma(r, 1.0 / 120.0, 1.0 / 24.0);
  p = fma(p, r, 1.0 / 6.0);
  p = fma(p, r, 0.5);
  p = fma(r * r, p, r);
  const double s = tab[n & 63];
  const double v = fma(s, p, s);
  return __hiloint2double(__double2hiint(v) + ((n >> 6) << 20), __double2loint(v));
}

// The variable behind node (a0, a1, a2): the node itself, or its mirror image in the first octant.
__device__ __forceinline__ int variable(int a0, int a1, int a2, int nd0, int nd1, int nd2, int octant) {
  if (!octant) return (a0 * nd1 + a1) * nd2 + a2;
  return (min(a0, nd0 - 1 - a0) * (nd1 / 2) + min(a1, nd1 - 1 - a1)) * (nd2 / 2) + min(a2, nd2 - 1 - a2);
}

// Average and projection.  Bound: the FP64 unit (one instruction of all elements of a 96^3 cell is 1.5 us):
// one multiply-add per node within the radius (13 in FCC at the default), 10 for the exponential and 6 more.
// Two library exponentials and FP64 clamps took 88 us on that cell, this 46 us.
// eb: exp(-beta).  small: beta < 690.
__global__ void k_project(const double* __restrict__ x, const DesignEntry* __restrict__ tab,
                          const int* __restrict__ cstart, int n0, int n1, int n2, int nd0, int nd1, int nd2, int sp, int octant,
                          double beta, double eb, int small, const double* __restrict__ exp2t, double* __restrict__ rho,
                          double* __restrict__ dmu) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)n0 * n1 * n2) return;
  const int l = (int)(e % n2), j = (int)((e / n2) % n1), i = (int)(e / ((long long)n1 * n2));
  const int b0 = i / sp, b1 = j / sp, b2 = l / sp;
  const int p = ((i - b0 * sp) * sp + (j - b1 * sp)) * sp + (l - b2 * sp);
  double mu = 0.0;
#pragma unroll 4
  for (int q = cstart[p]; q < cstart[p + 1]; ++q) {
    const DesignEntry t = tab[q];
    const int a0 = wrap(b0 + t.d0, nd0), a1 = wrap(b1 + t.d1, nd1), a2 = wrap(b2 + t.d2, nd2);
    mu = fma(t.w, x[variable(a0, a1, a2, nd0, nd1, nd2, octant)], mu);
  }
  // mu is a convex combination of values in [0, 1]: the clamps only remove rounding excursions
  // (a density 1 ulp above 1 would be flagged PC_EDOMAIN by pc_set_design)
  mu = clamp01(mu);
  const double em = small ? exp_tab(-beta * mu, exp2t) : exp(-beta * mu);
  rho[e] = clamp01(1.0 - em + mu * eb);
  dmu[e] = beta * em + eb;
}

__global__ void k_grad_mu(const double* __restrict__ g_rho, const double* __restrict__ dmu, long long ne,
                          double* __restrict__ gmu) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < ne) gmu[e] = g_rho[e] * dmu[e];
}

// dG/dphi_a = sum over the elements e that average node a of w_ea dG/drho_e drho_e/dmu_e.  DONE: g is
// dG/dmu_e already; it takes a pass over the elements but one FP64 instruction per node and element instead
// of two (96^3, FCC: 45 us in one launch, 28 us in two; below GRAD_PASS elements the launch costs more).
// OCTANT: eight threads of a warp take the eight images of a variable and add up their sums in order.
template <bool DONE, bool OCTANT>
__global__ void k_project_grad(const double* __restrict__ g, const double* __restrict__ dmu,
                               const DesignEntry* __restrict__ tab, const int* __restrict__ cstart, int nclass,
                               int n1, int n2, int nd0, int nd1, int nd2, int sp, double* __restrict__ gx) {
  const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = t0 < (long long)nd0 * nd1 * nd2;
  if (!OCTANT && !in) return;
  int a0, a1, a2;
  const int m = (int)(t0 & 7);
  if (OCTANT) {
    const int h1 = nd1 / 2, h2 = nd2 / 2;
    const long long v = in ? t0 >> 3 : 0;
    const int c = (int)(v % h2), b = (int)((v / h2) % h1), a = (int)(v / ((long long)h1 * h2));
    a0 = (m & 1) ? nd0 - 1 - a : a;
    a1 = (m & 2) ? nd1 - 1 - b : b;
    a2 = (m & 4) ? nd2 - 1 - c : c;
  } else {
    a2 = (int)(t0 % nd2);
    a1 = (int)((t0 / nd2) % nd1);
    a0 = (int)(t0 / ((long long)nd1 * nd2));
  }
  double s = 0.0;
  for (int p = 0; p < nclass; ++p) {
    const int p0 = p / (sp * sp), p1 = (p / sp) % sp, p2 = p % sp;
#pragma unroll 4
    for (int q = cstart[p]; q < cstart[p + 1]; ++q) {
      const DesignEntry t = tab[q];
      const int b0 = wrap(a0 - t.d0, nd0), b1 = wrap(a1 - t.d1, nd1), b2 = wrap(a2 - t.d2, nd2);
      const int e = ((sp * b0 + p0) * n1 + (sp * b1 + p1)) * n2 + (sp * b2 + p2);
      s = fma(t.w, DONE ? g[e] : g[e] * dmu[e], s);
    }
  }
  if (OCTANT) {
    double f = 0.0;
    for (int i = 0; i < 8; ++i) f += __shfl_sync(0xffffffffu, s, i, 8);
    if (in && m == 0) gx[t0 >> 3] = f;
  } else {
    gx[t0] = s;
  }
}
constexpr long long GRAD_PASS = 1 << 18;

// Whether a call on stream s (identity id) may write the map's gmu: the last launch that reads it is done, or ahead
// on the same stream.  Gradients of one projection (objective and constraint) may be carried back on several
// streams at once, and a captured call replays whenever its graph is launched: these take the kernel without
// gmu, which gives the same bits.
bool gmu_claim(pc_design* d, cudaStream_t s, unsigned long long* id) {
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  bool ok = cudaStreamIsCapturing(s, &capture) == cudaSuccess && capture == cudaStreamCaptureStatusNone &&
            cudaStreamGetId(s, id) == cudaSuccess;
  if (ok && d->gmu_used && d->gmu_stream != *id) {
    // the event is none of any capture's, so the query disturbs none, whatever another thread records
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    ok = cudaThreadExchangeStreamCaptureMode(&mode) == cudaSuccess;
    if (ok) {
      ok = cudaEventQuery(d->gmu_read) == cudaSuccess;
      cudaThreadExchangeStreamCaptureMode(&mode);
    }
  }
  if (!ok) cudaGetLastError();
  return ok;
}

void lattice_columns(int lat, double a, double A[9]) {
  // columns a_1, a_2, a_3 (A[r*3+c] = component r of a_c)
  static const double P[3][3][3] = {{{1, 0, 0}, {0, 1, 0}, {0, 0, 1}},
                                    {{-0.5, 0.5, 0.5}, {0.5, -0.5, 0.5}, {0.5, 0.5, -0.5}},
                                    {{0, 0.5, 0.5}, {0.5, 0, 0.5}, {0.5, 0.5, 0}}};
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) A[r * 3 + c] = a * P[lat][c][r];
}

}  // namespace

extern "C" int pc_design_create(const pc_params* cell, const pc_design_params* dp, pc_design** out) {
  if (!out) return PC_EINVAL;
  *out = nullptr;
  if (!cell || !dp) return PC_EINVAL;
  if (cell->lattice < PC_SC || cell->lattice > PC_FCC || !(cell->a > 0) || !std::isfinite(cell->a)) return PC_EINVAL;
  if (dp->spacing != 1 && dp->spacing != 2) return PC_EINVAL;
  if (!(dp->radius > 0) || !std::isfinite(dp->radius)) return PC_EINVAL;
  if (dp->octant != 0 && dp->octant != 1) return PC_EINVAL;
  if (dp->octant && cell->lattice != PC_SC) return PC_EINVAL;
  const int sp = dp->spacing;
  int n[3], nd[3];
  for (int i = 0; i < 3; ++i) {
    n[i] = cell->n[i];
    if (n[i] < 1 || n[i] > 256 || n[i] % sp) return PC_EINVAL;
    nd[i] = n[i] / sp;
    if (dp->octant && nd[i] % 2) return PC_EINVAL;
  }
  double A[9];
  lattice_columns(cell->lattice, cell->a, A);
  // reciprocal vectors b_i (rows of A^-1).  A node at offset d along axis i has fractional offset
  // f_i = (sp d + sp/2 - p_i - 1/2) / n_i from the element and lies at least |f_i| / |b_i| away, so
  // only |sp d| < r n_i |b_i| + (sp - 1)/2 can fall within the radius: |d| <= R_i below.
  const double det = A[0] * (A[4] * A[8] - A[5] * A[7]) - A[1] * (A[3] * A[8] - A[5] * A[6]) +
                     A[2] * (A[3] * A[7] - A[4] * A[6]);
  const double inv[9] = {(A[4] * A[8] - A[5] * A[7]) / det, (A[2] * A[7] - A[1] * A[8]) / det,
                         (A[1] * A[5] - A[2] * A[4]) / det, (A[5] * A[6] - A[3] * A[8]) / det,
                         (A[0] * A[8] - A[2] * A[6]) / det, (A[2] * A[3] - A[0] * A[5]) / det,
                         (A[3] * A[7] - A[4] * A[6]) / det, (A[1] * A[6] - A[0] * A[7]) / det,
                         (A[0] * A[4] - A[1] * A[3]) / det};
  int R[3];
  for (int i = 0; i < 3; ++i) {
    const double bl = std::sqrt(inv[i * 3] * inv[i * 3] + inv[i * 3 + 1] * inv[i * 3 + 1] + inv[i * 3 + 2] * inv[i * 3 + 2]);
    R[i] = (int)std::floor((dp->radius * n[i] * bl + 0.5 * (sp - 1)) / sp);
    if (2 * R[i] + 1 > nd[i]) return PC_EINVAL;  // the radius reaches a node's periodic image
  }
  // weight table per parity class
  const int nclass = sp * sp * sp;
  std::vector<DesignEntry> tab;
  std::vector<int> cstart(nclass + 1, 0);
  for (int p = 0; p < nclass; ++p) {
    const int pc[3] = {p / (sp * sp), (p / sp) % sp, p % sp};
    const size_t first = tab.size();
    double tot = 0.0;
    for (int d0 = -R[0]; d0 <= R[0]; ++d0)
      for (int d1 = -R[1]; d1 <= R[1]; ++d1)
        for (int d2 = -R[2]; d2 <= R[2]; ++d2) {
          const int d[3] = {d0, d1, d2};
          double best = 1e300;
          for (int s0 = -1; s0 <= 1; ++s0)
            for (int s1 = -1; s1 <= 1; ++s1)
              for (int s2 = -1; s2 <= 1; ++s2) {
                const int sh[3] = {s0, s1, s2};
                double f[3], x[3] = {0, 0, 0};
                for (int ax = 0; ax < 3; ++ax) f[ax] = (sp * d[ax] + 0.5 * sp - pc[ax] - 0.5) / n[ax] + sh[ax];
                for (int r = 0; r < 3; ++r)
                  for (int c = 0; c < 3; ++c) x[r] += A[r * 3 + c] * f[c];
                best = std::fmin(best, std::sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]));
              }
          const double w = dp->radius - best;
          if (w > 0) {
            tab.push_back(DesignEntry{d0, d1, d2, w});
            tot += w;
          }
        }
    if (!(tot > 0)) return PC_EINVAL;  // an element sees no node within the radius
    for (size_t q = first; q < tab.size(); ++q) tab[q].w /= tot;
    cstart[p + 1] = (int)tab.size();
  }
  pc_design* d = new (std::nothrow) pc_design();
  if (!d) return PC_ENOMEM;
  memcpy(d->n, n, sizeof(n));
  memcpy(d->nd, nd, sizeof(nd));
  d->spacing = sp;
  d->octant = dp->octant;
  d->ne = (long long)n[0] * n[1] * n[2];
  d->nnodes = (long long)nd[0] * nd[1] * nd[2];
  d->nvars = dp->octant ? d->nnodes / 8 : d->nnodes;
  d->nclass = nclass;
  // [exp2t | table | class_start] as staged on the host, then dmu and gmu
  const size_t ts = sizeof(DesignEntry) * tab.size(), cs = sizeof(int) * (nclass + 1);
  const size_t head = (64 * sizeof(double) + ts + cs + 255) / 256 * 256;
  const size_t field = (sizeof(double) * d->ne + 255) / 256 * 256;
  unsigned char* base = nullptr;
  if (cudaMalloc(&base, head + (d->ne < GRAD_PASS ? 1 : 2) * field) != cudaSuccess) {
    cudaGetLastError();
    pc_design_destroy(d);
    return PC_ENOMEM;
  }
  d->exp2t = (double*)base;
  d->table = (DesignEntry*)(base + 64 * sizeof(double));
  d->class_start = (int*)(base + 64 * sizeof(double) + ts);
  d->dmu = (double*)(base + head);
  if (d->ne >= GRAD_PASS) {
    if (cudaEventCreateWithFlags(&d->gmu_read, cudaEventDisableTiming) != cudaSuccess) {
      pc_design_destroy(d);
      return PC_ECUDA;
    }
    d->gmu = (double*)(base + head + field);
  }
  std::vector<unsigned char> stage(head, 0);
  for (int j = 0; j < 64; ++j) ((double*)stage.data())[j] = std::exp2(j / 64.0);
  memcpy(stage.data() + 64 * sizeof(double), tab.data(), ts);
  memcpy(stage.data() + 64 * sizeof(double) + ts, cstart.data(), cs);
  if (cudaMemcpy(base, stage.data(), head, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemset(d->dmu, 0, sizeof(double) * d->ne) != cudaSuccess) {
    pc_design_destroy(d);
    return PC_ECUDA;
  }
  *out = d;
  return PC_OK;
}

extern "C" long long pc_design_nvars(const pc_design* d) { return d ? d->nvars : -1; }

extern "C" int pc_design_project(pc_design* d, const double* x, double beta, double* rho, void* stream) {
  if (!d || !x || !rho || !(beta > 0) || !std::isfinite(beta)) return PC_EINVAL;
  cudaGetLastError();
  cudaStream_t s = (cudaStream_t)stream;
  k_project<<<cdiv(d->ne, 256), 256, 0, s>>>(x, d->table, d->class_start, d->n[0], d->n[1], d->n[2], d->nd[0],
                                             d->nd[1], d->nd[2], d->spacing, d->octant, beta, std::exp(-beta),
                                             beta < 690.0, d->exp2t, rho, d->dmu);
  PC_LAUNCH_CHECK();
  return PC_OK;
}

extern "C" int pc_design_backprop(pc_design* d, const double* g_rho, double* g_x, void* stream) {
  if (!d || !g_rho || !g_x) return PC_EINVAL;
  cudaGetLastError();
  cudaStream_t s = (cudaStream_t)stream;
  const double* g = g_rho;
  std::unique_lock<std::mutex> lock(d->gmu_lock, std::defer_lock);
  double* gmu = nullptr;
  unsigned long long id = 0;
  if (d->ne >= GRAD_PASS) {
    lock.lock();
    if (d->gmu && gmu_claim(d, s, &id)) std::swap(gmu, d->gmu);  // given back once its event is recorded
  }
  if (gmu) {
    k_grad_mu<<<cdiv(d->ne, 256), 256, 0, s>>>(g_rho, d->dmu, d->ne, gmu);
    PC_LAUNCH_CHECK();
    g = gmu;
  }
  auto kernel = d->octant ? (gmu ? k_project_grad<true, true> : k_project_grad<false, true>)
                          : (gmu ? k_project_grad<true, false> : k_project_grad<false, false>);
  kernel<<<cdiv(d->nnodes, 128), 128, 0, s>>>(g, d->dmu, d->table, d->class_start, d->nclass, d->n[1], d->n[2], d->nd[0],
                                              d->nd[1], d->nd[2], d->spacing, g_x);
  PC_LAUNCH_CHECK();
  if (gmu) {
    PC_CUDA_TRY(cudaEventRecord(d->gmu_read, s));
    d->gmu_stream = id;
    d->gmu_used = true;
    d->gmu = gmu;
  }
  return PC_OK;
}

extern "C" void pc_design_destroy(pc_design* d) {
  if (!d) return;
  if (d->exp2t) cudaFree(d->exp2t);
  if (d->gmu_read) cudaEventDestroy(d->gmu_read);
  delete d;
}

// C ABI, context and host orchestration of the band + adjoint path.
//
// Per design (pc_set_design): SIMP interpolation, structure factors, Toeplitz operators
// and the two inverse compliance operators (setup.cu).
// Per band evaluation (pc_bands): a batched block preconditioned eigensolver over all
// k at once (one independent projected problem per k), followed by one FP64
// Rayleigh-Ritz step that also yields the FP64 stress coefficients for the adjoint.
// PC_FP64 runs the block iteration in FP64; PC_MIXED runs it with FP32 vectors and
// the split-BF16 tensor-core operator (gemm_tc.cu), then refines in FP64.
// Per objective (pc_gap_and_grad): gap and weights, field synthesis and the weighted
// per-voxel reduction (adjoint.cu).
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <utility>
#include <atomic>
#include <mutex>
#include <thread>
#include <type_traits>
#include <vector>
#include "kernels.h"
#include "gemm_tc.h"
#include "launch_rules.h"


std::atomic<long long> g_pc_launches{0};

// Per-phase device timing (pc_set_profiling): event pairs recorded on the caller's stream.
enum { PH_RR_GEMM = 0, PH_ITER_APPLY = 1, PH_SMALL = 2, PH_GRAD = 3, PH_GRAM = 4, PH_UPDATE = 5, PH_LOOP = 6,
       PH_FINAL = 7, PH_IDLE = 8, PH_COUNT = 9 };
// Smallest k group worth its own stream, and the most groups (mixed form, see pc_bands).
constexpr int kSplitMinK = 16;
constexpr int kMaxGroups = 6;

struct EventPair {
  cudaEvent_t a, b;
  int phase;
  double flops;
  double bytes;
};

struct pc_ctx {
  pc_params prm;
  int N, M2, L, ne, m, nb;
  int nk = 0;
  double A[9], Tm[9], V, ve;
  double lref, sO, sA, cA;  // lambda scale, Omega scale, operator scale, (2 pi)^2 V^2 / sA
  Geom geom;
  MaterialConsts mc;
  PrecRef pr;
  bool have_design = false, have_bands = false, have_grad = false;
  int warm = 0;                  // pc_set_warm_start: start from the last final Ritz block
  bool warm_ready = false;       // Th holds a final block of the current k-points
  bool import_pending = false;   // pc_import_block: use Th as the start block of the next pc_bands
  int iterations = 0, unconv = 0;
  double max_res = 0.0;
  float ms_setup = 0.f, ms_bands = 0.f, ms_grad = 0.f;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;            // pc_bands
  cudaEvent_t ev_s0 = nullptr, ev_s1 = nullptr;        // pc_set_design
  cudaEvent_t ev_g0 = nullptr, ev_g1 = nullptr;        // pc_gap_and_grad
  bool have_grad_events = false;
  int* h_count = nullptr;   // pinned, 4 per k group (OpenSet::count)
  // per-design (FP64)
  double *fields = nullptr, *dchi = nullptr, *chi = nullptr, *chi_mean = nullptr, *dfc = nullptr;
  double2 *t1 = nullptr, *t2s = nullptr, *sfac = nullptr, *T = nullptr, *W = nullptr, *gj = nullptr;
  float2 *Wf = nullptr, *Tf = nullptr;  // scaled FP32 W1, W2 and T_rho, T_f1, T_f2 (mixed form without a tensor-core plan)
  bool f32_ready = false;               // they are of the current design
  double* prec_ref = nullptr;           // preconditioner reference medium, 3 values per k group
  int* status = nullptr;
  double* small_flops = nullptr;  // device: algorithmic flops of the FP32 projected problems while profiling
  double sig_scale = 1, w_scale = 1;  // powers of two: the final step's stresses and the adjoint's weights in FP32's range
  double grad_flops_per_pair = 0;  // algorithmic flops of the adjoint per weighted (k, band)
  // per k-set
  double* Q = nullptr;
  void* blk[15] = {nullptr};     // X AX OX W AW OW P AP OP Xn AXn OXn Pn APn OPn (R precision)
  void *E = nullptr, *S = nullptr;  // strain / stress stacks (R precision)
  void *gpart = nullptr, *GA = nullptr, *GO = nullptr, *Cc = nullptr, *Ct = nullptr;
  void* lam = nullptr;           // nk*m (R)
  unsigned char* sr_scratch = nullptr;  // scratch of the projected problems in flight (small_rr.cu, small_rr64.cu)
  long long sr_stride = 0;              // bytes per problem
  double *rnorm = nullptr;
  int *active = nullptr, *kdone = nullptr, *kdone_f = nullptr;
  int *open_k = nullptr, *open_v = nullptr, *open_pos = nullptr, *fresh_k = nullptr, *d_count = nullptr;  // OpenSet, per k group at its k0
  double* stall_best = nullptr;  // per k: best worst-wanted residual so far (stagnation test)
  int* stall_since = nullptr;     // per k: iterations since that best
  // FP64 Rayleigh-Ritz and adjoint
  double2 *Xd = nullptr, *AXd = nullptr, *OXd = nullptr, *Ed = nullptr, *Sd = nullptr, *Th = nullptr, *St = nullptr;
  double2 *gpartd = nullptr, *GAd = nullptr, *GOd = nullptr, *Cd = nullptr;
  double *lamd = nullptr, *lam_nd = nullptr, *rnormd = nullptr;
  int* actived = nullptr;
  double *weights = nullptr;
  int *pairs = nullptr, *npairs = nullptr;
  double2* adj_t2 = nullptr;
  double* adj_part = nullptr;  // chunk sums of the adjoint's reduction
  double2* adj_ph = nullptr;  // phases of the adjoint's synthesis (room for FP64)
  float4* Kf = nullptr;  // FP32 wavevectors of the k-points, [k][N] (mixed form)
  TcPlan* tc = nullptr;
  TcPlan* tcg[kMaxGroups] = {};  // workspaces of k groups 1.. (operators shared with tc)
  OzPlan* oz = nullptr;          // sliced FP64-accurate operators of the final Rayleigh-Ritz step (mixed form)
  OzPlan* ozg[kMaxGroups] = {};  // right-hand-side workspaces of k groups 1.. (operators shared with oz)
  bool oz_ready = false;         // oz holds the slices of the current design
  cudaStream_t sk[kMaxGroups] = {};  // non-blocking streams of the k groups
  cudaEvent_t ev_fork = nullptr, ev_join[kMaxGroups] = {};
  int split = 1;                // PC_SPLIT=0: the block iteration of the mixed form on one stream
  int groups = 2;               // k groups run concurrently (PC_KGROUPS, 2..kMaxGroups)
  std::mutex ph_mu;             // profiling records from the two k-half threads
  bool tc_ready = false;        // tensor-core operands prepared for the current design
  int debug = 0;  // PC_DEBUG=1 prints the residual history of the block iteration to stderr
  int profiling = 0;
  std::vector<EventPair> ev_used, ev_free;
  double ph_ms[PH_COUNT] = {};
  double ph_flops[PH_COUNT] = {};
  double ph_bytes[PH_COUNT] = {};
  long long ph_count[PH_COUNT] = {};
  long long launch_base = 0;
  unsigned long long seed = 0;  // PC_INIT_SEED: offset of the start-block perturbation
  int refresh = 40;             // iterations between recomputations of A X, Omega X (PC_REFRESH)
};

// Number of k groups of the mixed form's block iteration for nk k-points (1: one stream).
static int kgroups(const pc_ctx* c, int nk) {
  if (!c->split || c->prm.precision != PC_MIXED) return 1;
  return std::max(1, std::min(c->groups, nk / kSplitMinK));
}

// First of the projected problems' scratch slots of group g of `groups` (g = groups: all of them; the set as one group
// needs no more).
static long long rr_first(int nk, int groups, int g) {
  long long first = 0;
  for (int h = 0; h < g; ++h)
    first += rr_problems_per_launch((long long)nk * (h + 1) / groups - (long long)nk * h / groups, device_sms());
  return first;
}

// Opens a timed phase on stream s (no-op unless profiling); returns the slot index or -1.
static int ph_begin(pc_ctx* c, int phase, double flops, cudaStream_t s, double bytes = 0.0) {
  if (!c->profiling) return -1;
  std::lock_guard<std::mutex> lk(c->ph_mu);
  EventPair e;
  if (!c->ev_free.empty()) {
    e = c->ev_free.back();
    c->ev_free.pop_back();
  } else {
    if (cudaEventCreate(&e.a) != cudaSuccess || cudaEventCreate(&e.b) != cudaSuccess) return -1;
  }
  e.phase = phase;
  e.flops = flops;
  e.bytes = bytes;
  cudaEventRecord(e.a, s);
  c->ev_used.push_back(e);
  return (int)c->ev_used.size() - 1;
}
static void ph_end(pc_ctx* c, int slot, cudaStream_t s) {
  if (slot < 0) return;
  std::lock_guard<std::mutex> lk(c->ph_mu);
  cudaEventRecord(c->ev_used[slot].b, s);
}
// Folds finished event pairs into the sums (caller has synchronised).
static void ph_collect(pc_ctx* c) {
  for (auto& e : c->ev_used) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, e.a, e.b) == cudaSuccess) {
      c->ph_ms[e.phase] += ms;
      c->ph_flops[e.phase] += e.flops;
      c->ph_bytes[e.phase] += e.bytes;
      c->ph_count[e.phase] += 1;
    }
    c->ev_free.push_back(e);
  }
  c->ev_used.clear();
  cudaGetLastError();
}

static const char* kErr[] = {"PC_OK", "PC_EINVAL", "PC_EALIAS", "PC_ENOMEM", "PC_ECUDA",
                             "PC_ESTATE", "PC_ENOCONV", "PC_EDOMAIN", "PC_ETIMEOUT", "PC_ETOOBIG"};

extern "C" const char* pc_strerror(int code) {
  if (code < 0 || code > 9) return "PC_UNKNOWN";
  return kErr[code];
}

template <typename T> static int dalloc(T** p, size_t count) {
  *p = nullptr;
  if (count == 0) count = 1;
  if (cudaMalloc((void**)p, count * sizeof(T)) != cudaSuccess) {
    *p = nullptr;
    cudaGetLastError();
    return PC_ENOMEM;
  }
  return PC_OK;
}
template <typename T> static void dfree(T*& p) {
  if (p) cudaFree((void*)p);
  p = nullptr;
}

bool pc_material_ok(const pc_material& m) {
  return m.rho > 0 && m.E > 0 && m.nu > -1.0 && m.nu < 0.5 && std::isfinite(m.rho) && std::isfinite(m.E);
}

static void lattice_vectors(int lat, double a, double A[9]) {
  // columns a_1, a_2, a_3; A[r*3+c] = component r of a_c
  double P[3][3];
  if (lat == PC_SC) {
    double t[3][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}};
    memcpy(P, t, sizeof(P));
  } else if (lat == PC_BCC) {
    double t[3][3] = {{-0.5, 0.5, 0.5}, {0.5, -0.5, 0.5}, {0.5, 0.5, -0.5}};  // rows: a_1, a_2, a_3
    memcpy(P, t, sizeof(P));
  } else {
    double t[3][3] = {{0, 0.5, 0.5}, {0.5, 0, 0.5}, {0.5, 0.5, 0}};
    memcpy(P, t, sizeof(P));
  }
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) A[r * 3 + c] = a * P[c][r];
}

static double det3(const double m[9]) {
  return m[0] * (m[4] * m[8] - m[5] * m[7]) - m[1] * (m[3] * m[8] - m[5] * m[6]) + m[2] * (m[3] * m[7] - m[4] * m[6]);
}

// T = A^{-T}: b_i . a_j = delta_ij, T row-major with K = T (Q + g)
static void reciprocal(const double A[9], double T[9]) {
  double d = det3(A);
  double inv[9];
  inv[0] = (A[4] * A[8] - A[5] * A[7]) / d;
  inv[1] = (A[2] * A[7] - A[1] * A[8]) / d;
  inv[2] = (A[1] * A[5] - A[2] * A[4]) / d;
  inv[3] = (A[5] * A[6] - A[3] * A[8]) / d;
  inv[4] = (A[0] * A[8] - A[2] * A[6]) / d;
  inv[5] = (A[2] * A[3] - A[0] * A[5]) / d;
  inv[6] = (A[3] * A[7] - A[4] * A[6]) / d;
  inv[7] = (A[1] * A[6] - A[0] * A[7]) / d;
  inv[8] = (A[0] * A[4] - A[1] * A[3]) / d;
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 3; ++c) T[r * 3 + c] = inv[c * 3 + r];
}

static void lame(const pc_material& m, double* lam, double* mu) {
  *mu = m.E / (2.0 * (1.0 + m.nu));
  *lam = m.E * m.nu / ((1.0 + m.nu) * (1.0 - 2.0 * m.nu));
}

static void free_kset(pc_ctx* c) {
  dfree(c->Q);
  for (auto& b : c->blk) { if (b) cudaFree(b); b = nullptr; }
  if (c->E) cudaFree(c->E); c->E = nullptr;
  if (c->S) cudaFree(c->S); c->S = nullptr;
  void** vs[] = {&c->gpart, &c->GA, &c->GO, &c->Cc, &c->Ct, &c->lam};
  for (auto v : vs) { if (*v) cudaFree(*v); *v = nullptr; }
  dfree(c->sr_scratch);
  dfree(c->open_k);  // and with it:
  c->fresh_k = c->kdone = c->kdone_f = c->stall_since = c->open_v = c->open_pos = c->active = c->actived = nullptr;
  c->d_count = c->pairs = c->npairs = nullptr;
  dfree(c->GAd);  // and with it:
  c->GOd = c->Cd = nullptr;
  c->rnorm = c->lamd = c->rnormd = c->lam_nd = c->weights = c->stall_best = nullptr;
  dfree(c->Xd); dfree(c->AXd); dfree(c->OXd); dfree(c->Ed); dfree(c->Sd); dfree(c->Th); dfree(c->St);
  dfree(c->gpartd); dfree(c->adj_t2); dfree(c->adj_part); dfree(c->Kf);
  for (auto& t : c->tcg)
    if (t) { tc_plan_destroy(t); t = nullptr; }
  if (c->tc) { tc_plan_destroy(c->tc); c->tc = nullptr; }
  for (auto& o : c->ozg)
    if (o) { oz_plan_destroy(o); o = nullptr; }
  if (c->oz) { oz_plan_destroy(c->oz); c->oz = nullptr; }
  c->oz_ready = false;
  c->nk = 0;
  c->have_bands = false;
  c->have_grad = false;
  c->warm_ready = false;
  c->import_pending = false;
}

extern "C" void pc_destroy(pc_ctx* c) {
  if (!c) return;
  free_kset(c);
  dfree(c->fields); dfree(c->dchi); dfree(c->chi); dfree(c->chi_mean); dfree(c->dfc);
  dfree(c->t1); dfree(c->t2s); dfree(c->sfac); dfree(c->T); dfree(c->W); dfree(c->gj);
  dfree(c->Wf); dfree(c->Tf); dfree(c->status); dfree(c->small_flops); dfree(c->adj_ph);
  if (c->ev0) cudaEventDestroy(c->ev0);
  if (c->ev1) cudaEventDestroy(c->ev1);
  for (cudaEvent_t e : {c->ev_s0, c->ev_s1, c->ev_g0, c->ev_g1})
    if (e) cudaEventDestroy(e);
  for (auto& e : c->ev_used) { cudaEventDestroy(e.a); cudaEventDestroy(e.b); }
  for (auto& e : c->ev_free) { cudaEventDestroy(e.a); cudaEventDestroy(e.b); }
  if (c->h_count) cudaFreeHost(c->h_count);
  for (int i = 0; i < kMaxGroups; ++i) {
    if (c->sk[i]) cudaStreamDestroy(c->sk[i]);
    if (c->ev_join[i]) cudaEventDestroy(c->ev_join[i]);
  }
  if (c->ev_fork) cudaEventDestroy(c->ev_fork);
  delete c;
}

extern "C" int pc_create(const pc_params* p, pc_ctx** out) {
  if (!out) return PC_EINVAL;
  *out = nullptr;
  if (!p) return PC_EINVAL;
  if (p->lattice < PC_SC || p->lattice > PC_FCC) return PC_EINVAL;
  if (!(p->a > 0) || !std::isfinite(p->a)) return PC_EINVAL;
  if (p->M < 1 || p->M > 5) return PC_EINVAL;
  for (int i = 0; i < 3; ++i)
    if (p->n[i] < 1 || p->n[i] > 256) return PC_EINVAL;
  if (!pc_material_ok(p->phase0) || !pc_material_ok(p->phase1)) return PC_EINVAL;
  if (!(p->penal >= 1.0) || !std::isfinite(p->penal)) return PC_EINVAL;
  if (p->precision != PC_FP64 && p->precision != PC_MIXED) return PC_EINVAL;
  if (p->tol < 0 || p->max_iter < 0) return PC_EINVAL;
  if (p->law != PC_LAW_COMPLIANCE && p->law != PC_LAW_YOUNG) return PC_EINVAL;
  const int M2 = 2 * p->M + 1;
  const int N = M2 * M2 * M2;
  if (p->nbands < 1 || p->nbands > 24 || p->nbands > N) return PC_EINVAL;
  for (int i = 0; i < 3; ++i)
    if (p->n[i] < M2) return PC_EALIAS;

  pc_ctx* c = new (std::nothrow) pc_ctx();
  if (!c) return PC_ENOMEM;
  c->prm = *p;
  {
    const char* dbg = getenv("PC_DEBUG");
    c->debug = (dbg && dbg[0] == '1') ? 1 : 0;
    const char* rf = getenv("PC_REFRESH");
    if (rf && atoi(rf) > 0) c->refresh = atoi(rf);
    const char* sd = getenv("PC_INIT_SEED");
    c->seed = sd ? strtoull(sd, nullptr, 10) : 0ull;
    const char* sp = getenv("PC_SPLIT");
    c->split = (sp && sp[0] == '0') ? 0 : 1;
    const char* kg = getenv("PC_KGROUPS");
    if (kg && atoi(kg) >= 2 && atoi(kg) <= kMaxGroups) c->groups = atoi(kg);
  }
  // Default residual targets: 1e-8 for the FP64 form; 3e-4 for the FP32 iteration of the mixed
  // form, whose final FP64 Rayleigh-Ritz step makes eigenvalue errors quadratic in the residual
  // (measured on the FCC N = 729 designs: frequencies within 1e-8 and gradients within 1.4e-5
  // of the FP64 form at 4e-4, 20 % fewer iterations than at 1e-4).
  if (c->prm.tol == 0) c->prm.tol = (p->precision == PC_FP64) ? 1e-8 : 3e-4;
  if (c->prm.max_iter == 0) c->prm.max_iter = (p->precision == PC_FP64) ? 600 : 400;
  c->M2 = M2;
  c->N = N;
  c->L = 4 * p->M + 1;
  c->ne = p->n[0] * p->n[1] * p->n[2];
  c->nb = p->nbands;
  {
    // guard vectors beyond the wanted bands: 3 in the mixed form (smaller projected problems,
    // the same iteration count there), 4 in the FP64 form (fewer iterations); PC_GUARD overrides
    const char* gv = getenv("PC_GUARD");
    const int guard = (gv && atoi(gv) >= 1 && atoi(gv) <= 8) ? atoi(gv) : (p->precision == PC_MIXED ? 3 : 4);
    c->m = std::min(std::min(p->nbands + guard, 24), N);
  }
  lattice_vectors(p->lattice, p->a, c->A);
  reciprocal(c->A, c->Tm);
  c->V = std::fabs(det3(c->A));
  c->ve = c->V / c->ne;
  const double two_pi = 2.0 * M_PI;
  c->lref = two_pi * two_pi * p->phase1.E / (p->phase1.rho * p->a * p->a);
  c->sO = c->V * p->phase1.rho;
  c->sA = c->lref * c->sO;
  c->cA = two_pi * two_pi * c->V * c->V / c->sA;
  {
    // The stress coefficients sigma of a normalised eigenvector satisfy (2 pi V)^2 V f |sigma|^2 / sO = lambda (f a
    // compliance modulus), and the gradient sums w |sigma|^2 with w = dG/dlambda.  In SI sigma goes as a^-4 and its
    // square leaves FP32 for cells of a millimetre; scaled to |sigma|^2 = lambda / lref, and w by lref, both
    // factors are nondimensional.  Exact, being powers of two.
    const double f = (1.0 + p->phase1.nu) / p->phase1.E;
    const double v = two_pi * c->V * std::sqrt(f * c->V / c->sO) / std::sqrt(c->lref);
    if (std::isnormal(v) && std::isnormal(c->lref)) {
      c->sig_scale = std::ldexp(1.0, std::ilogb(v));
      c->w_scale = std::ldexp(1.0, std::ilogb(c->lref));
    }
  }
  memcpy(c->geom.T, c->Tm, sizeof(c->Tm));
  c->geom.M = p->M;
  c->geom.N = N;
  c->mc.law = p->law;
  c->mc.E0 = p->phase0.E;
  c->mc.E1 = p->phase1.E;
  c->mc.nu0 = p->phase0.nu;
  c->mc.nu1 = p->phase1.nu;
  c->mc.penal = p->penal;
  c->mc.rho0 = p->phase0.rho;
  c->mc.rho1 = p->phase1.rho;
  c->mc.f1_0 = (1.0 - 2.0 * p->phase0.nu) / p->phase0.E;
  c->mc.f1_1 = (1.0 - 2.0 * p->phase1.nu) / p->phase1.E;
  c->mc.f2_0 = (1.0 + p->phase0.nu) / p->phase0.E;
  c->mc.f2_1 = (1.0 + p->phase1.nu) / p->phase1.E;
  lame(p->phase0, &c->pr.lam0, &c->pr.mu0);
  lame(p->phase1, &c->pr.lam1, &c->pr.mu1);
  c->pr.rho0 = p->phase0.rho;
  c->pr.rho1 = p->phase1.rho;
  c->pr.f1_0 = (1.0 - 2.0 * p->phase0.nu) / p->phase0.E;
  c->pr.f1_1 = (1.0 - 2.0 * p->phase1.nu) / p->phase1.E;
  c->pr.f2_0 = (1.0 + p->phase0.nu) / p->phase0.E;
  c->pr.f2_1 = (1.0 + p->phase1.nu) / p->phase1.E;
  {
    // Reference medium of the preconditioner at the mean chi: moduli between the material's with the mean
    // compliance (PC_PREC_REF=1) and with the mean Lame constants (0), their geometric mean; its shift is
    // PC_PREC_SHIFT times half the mass term rho sigma.  The iterations depend little on either: for shifts
    // of 0.04 to 0.5 and the three media within 10 % on level sets and 25 % on spheres (M = 2, 3).
    const char* rm = getenv("PC_PREC_REF");
    c->pr.ref_mode = (rm && rm[0] == '0') ? 0 : ((rm && rm[0] == '1') ? 1 : 2);
    const char* sh = getenv("PC_PREC_SHIFT");
    c->pr.shift_scale = (sh && atof(sh) > 0) ? atof(sh) : 0.1;
  }
  {
    // adjoint per weighted (k, band): 9 fields synthesised along axis 2, axis 1 and axis 0 (inside the voxel
    // reduction), 4 M real multiply-adds for two mirrored values
    const double m2 = M2, n0 = p->n[0], n1 = p->n[1], n2 = p->n[2];
    c->grad_flops_per_pair = 4.0 * p->M * 9.0 * (m2 * m2 * n2 + m2 * n1 * n2 + n0 * n1 * n2);
  }
  c->pr.two_pi_sq_V_over_sA = two_pi * two_pi * c->V / c->sA;
  c->pr.half_lref_V_over_sA = 0.5 * c->lref * c->V / c->sA;

  const size_t NN = (size_t)N * N;
  const size_t ne = c->ne, L = c->L;
  int rc = PC_OK;
  rc |= dalloc(&c->fields, 3 * ne);
  rc |= dalloc(&c->dchi, ne);
  rc |= dalloc(&c->chi, ne);
  rc |= dalloc(&c->dfc, 2 * ne);
  rc |= dalloc(&c->chi_mean, 1);
  rc |= dalloc(&c->t1, 3 * (size_t)p->n[0] * p->n[1] * L);
  rc |= dalloc(&c->t2s, 3 * (size_t)p->n[0] * L * L);
  rc |= dalloc(&c->sfac, 3 * L * L * L);
  rc |= dalloc(&c->T, 3 * NN);
  rc |= dalloc(&c->W, 2 * NN);
  rc |= dalloc(&c->gj, (size_t)setup_gj_scratch(N));
  rc |= dalloc(&c->status, 1);
  rc |= dalloc(&c->small_flops, 1);
  // one allocation: the phases, then the reference media
  const size_t nph = (size_t)p->M * (p->n[0] + p->n[1] + p->n[2]);
  rc |= dalloc(&c->adj_ph, nph + (3 * (size_t)kMaxGroups + 1) / 2);
  if (c->adj_ph) c->prec_ref = (double*)(c->adj_ph + nph);
  if (p->precision == PC_MIXED) {
    rc |= dalloc(&c->Wf, 2 * NN);
    rc |= dalloc(&c->Tf, 3 * NN);
  }
  if (rc != PC_OK) { pc_destroy(c); return PC_ENOMEM; }
  if (cudaMemset(c->status, 0, sizeof(int)) != cudaSuccess || cudaMemset(c->small_flops, 0, sizeof(double)) != cudaSuccess ||
      cudaEventCreate(&c->ev0) != cudaSuccess || cudaEventCreate(&c->ev1) != cudaSuccess ||
      cudaEventCreate(&c->ev_s0) != cudaSuccess || cudaEventCreate(&c->ev_s1) != cudaSuccess ||
      cudaEventCreate(&c->ev_g0) != cudaSuccess || cudaEventCreate(&c->ev_g1) != cudaSuccess ||
      cudaMallocHost((void**)&c->h_count, 4 * kMaxGroups * sizeof(int)) != cudaSuccess ||
      cudaEventCreateWithFlags(&c->ev_fork, cudaEventDisableTiming) != cudaSuccess) {
    pc_destroy(c);
    return PC_ECUDA;
  }
  // done before any work of a caller's stream: pc_set_kpoints copies on the same (legacy) stream and waits
  if (launch_adj_phases(p->M, p->n, p->precision == PC_MIXED, c->adj_ph, 0) != PC_OK) {
    pc_destroy(c);
    return PC_ECUDA;
  }
  for (int i = 0; i < kMaxGroups; ++i) {
    if (cudaStreamCreateWithFlags(&c->sk[i], cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&c->ev_join[i], cudaEventDisableTiming) != cudaSuccess) {
      pc_destroy(c);
      return PC_ECUDA;
    }
  }
  *out = c;
  return PC_OK;
}

extern "C" int pc_set_kpoints(pc_ctx* c, const double* q, int nk) {
  // The wavevector index is a grid dimension (y) of several launches: at most 65535.
  if (!c || !q || nk < 1 || nk > PC_MAX_KPOINTS) return PC_EINVAL;
  free_kset(c);
  const int m = c->m, N = c->N, n3 = 3 * N;
  const size_t nvec = (size_t)nk * m;
  const size_t esz = (c->prm.precision == PC_FP64) ? sizeof(double2) : sizeof(float2);
  const size_t rsz = (c->prm.precision == PC_FP64) ? sizeof(double) : sizeof(float);
  int rc = PC_OK;
  rc |= dalloc(&c->Q, 3 * (size_t)nk);
  if (c->prm.precision == PC_MIXED) rc |= dalloc(&c->Kf, (size_t)nk * N);
  for (auto& b : c->blk)
    if (cudaMalloc(&b, nvec * n3 * esz) != cudaSuccess) { b = nullptr; rc = PC_ENOMEM; }
  if (cudaMalloc(&c->E, 6 * nvec * N * esz) != cudaSuccess) { c->E = nullptr; rc = PC_ENOMEM; }
  if (cudaMalloc(&c->S, 6 * nvec * N * esz) != cudaSuccess) { c->S = nullptr; rc = PC_ENOMEM; }
  const size_t g = (size_t)nk * 72 * 72;
  if (cudaMalloc(&c->gpart, 8 * g * esz) != cudaSuccess) { c->gpart = nullptr; rc = PC_ENOMEM; }
  if (cudaMalloc(&c->GA, g * esz) != cudaSuccess) { c->GA = nullptr; rc = PC_ENOMEM; }
  if (cudaMalloc(&c->GO, g * esz) != cudaSuccess) { c->GO = nullptr; rc = PC_ENOMEM; }
  if (cudaMalloc(&c->Cc, g * esz) != cudaSuccess) { c->Cc = nullptr; rc = PC_ENOMEM; }
  if (cudaMalloc(&c->Ct, g * esz) != cudaSuccess) { c->Ct = nullptr; rc = PC_ENOMEM; }
  if (cudaMalloc(&c->lam, nvec * rsz) != cudaSuccess) { c->lam = nullptr; rc = PC_ENOMEM; }
  // FP32 problems of up to 3m columns and the FP64 ones of m of the final step, or FP64 ones of up to 3m
  c->sr_stride = c->prm.precision == PC_MIXED ? std::max(small_rr32_scratch(3 * m), small_rr64_scratch(m))
                                              : small_rr64_scratch(3 * m);
  const int groups = kgroups(c, nk);
  rc |= dalloc(&c->sr_scratch, (size_t)rr_first(nk, groups, groups) * c->sr_stride);
  // The small arrays in two allocations (25 us each).  [open_k | fresh_k | kdone | kdone_f | stall_since] per k,
  // [open_v | open_pos | active | actived] per vector, d_count, pairs per (k, band), npairs:
  const size_t nkb = (size_t)nk * c->nb;
  rc |= dalloc(&c->open_k, 5 * (size_t)nk + 4 * nvec + 4 * (size_t)kMaxGroups + nkb + 1);
  if (c->open_k) {
    c->fresh_k = c->open_k + nk;
    c->kdone = c->fresh_k + nk;
    c->kdone_f = c->kdone + nk;
    c->stall_since = c->kdone_f + nk;
    c->open_v = c->stall_since + nk;
    c->open_pos = c->open_v + nvec;
    c->active = c->open_pos + nvec;
    c->actived = c->active + nvec;
    c->d_count = c->actived + nvec;
    c->pairs = c->d_count + 4 * kMaxGroups;
    c->npairs = c->pairs + nkb;
  }
  // [GAd | GOd | Cd] m x m complex per k, then [rnorm | lamd | rnormd] per vector, [lam_nd | weights] per (k, band),
  // stall_best per k
  const size_t nmm = (size_t)nk * m * m;
  rc |= dalloc(&c->GAd, 3 * nmm + (3 * nvec + 2 * nkb + nk + 1) / 2);
  if (c->GAd) {
    c->GOd = c->GAd + nmm;
    c->Cd = c->GOd + nmm;
    c->rnorm = (double*)(c->Cd + nmm);
    c->lamd = c->rnorm + nvec;
    c->rnormd = c->lamd + nvec;
    c->lam_nd = c->rnormd + nvec;
    c->weights = c->lam_nd + nkb;
    c->stall_best = c->weights + nkb;
  }
  rc |= dalloc(&c->Xd, nvec * n3);
  rc |= dalloc(&c->AXd, nvec * n3);
  rc |= dalloc(&c->OXd, nvec * n3);
  rc |= dalloc(&c->Th, nvec * n3);
  rc |= dalloc(&c->Ed, 6 * nvec * N);
  rc |= dalloc(&c->Sd, 6 * nvec * N);
  rc |= dalloc(&c->St, 6 * nvec * N);
  rc |= dalloc(&c->gpartd, 8 * (size_t)nk * m * m);
  rc |= dalloc(&c->adj_t2, (size_t)nk * c->nb * 9 * c->M2 * c->prm.n[1] * c->prm.n[2]);
  rc |= dalloc(&c->adj_part, (size_t)kAdjChunksMax * 3 * c->prm.n[0] * c->prm.n[1] * c->prm.n[2]);
  if (rc == PC_OK && c->prm.precision == PC_MIXED) {
    c->tc = tc_plan_create(N, (int)nvec, c->status);
    c->tc_ready = false;
    if (!c->tc) rc = PC_ENOMEM;
    // the other k groups, run concurrently on streams of their own (run_split_iteration)
    const int ng = kgroups(c, nk);
    for (int g = 1; g < ng && c->tc; ++g) {
      const int gk = (int)(((long long)nk * (g + 1)) / ng - ((long long)nk * g) / ng);
      c->tcg[g] = tc_plan_create_sharing(c->tc, gk * m, c->status);
    }
    // the final Rayleigh-Ritz step's products: 6 strain stacks and 3 displacement columns per vector
    if (c->tc) {
      c->oz = oz_plan_create(N, 9 * (int)nvec, c->status, nullptr);
      for (int g = 1; g < ng && oz_available(c->oz); ++g) {
        const int gk = (int)(((long long)nk * (g + 1)) / ng - ((long long)nk * g) / ng);
        c->ozg[g] = oz_plan_create(N, 9 * gk * m, c->status, c->oz);
      }
      bool all = oz_available(c->oz);
      for (int g = 1; g < ng; ++g) all = all && oz_available(c->ozg[g]);
      if (!all) {  // keep the FP64 GEMM for this k-set
        for (auto& o : c->ozg)
          if (o) { oz_plan_destroy(o); o = nullptr; }
        if (c->oz) { oz_plan_destroy(c->oz); c->oz = nullptr; }
      }
    }
  }
  if (rc != PC_OK) { free_kset(c); return PC_ENOMEM; }
  if (cudaMemcpy(c->Q, q, 3 * sizeof(double) * nk, cudaMemcpyHostToDevice) != cudaSuccess) {
    free_kset(c);
    return PC_ECUDA;
  }
  if (c->Kf && (launch_kvec_table(c->geom, c->Q, nk, c->Kf, 0) != PC_OK || cudaStreamSynchronize(0) != cudaSuccess)) {
    free_kset(c);
    return PC_ECUDA;
  }
  c->nk = nk;
  return PC_OK;
}

extern "C" int pc_set_design(pc_ctx* c, const double* rho, void* stream) {
  if (!c || !rho) return PC_EINVAL;
  cudaGetLastError();  // launch checks below report only this call's launches
  cudaStream_t s = (cudaStream_t)stream;
  PC_CUDA_TRY(cudaEventRecord(c->ev_s0, s));
  SetupArgs a;
  a.rho = rho;
  a.n0 = c->prm.n[0]; a.n1 = c->prm.n[1]; a.n2 = c->prm.n[2];
  a.M = c->prm.M;
  a.V = c->V;
  a.mc = c->mc;
  a.fields = c->fields; a.dchi = c->dchi; a.chi = c->chi; a.chi_mean = c->chi_mean; a.dfc = c->dfc;
  a.t1 = c->t1; a.t2 = c->t2s; a.sfac = c->sfac; a.T = c->T; a.W = c->W;
  a.gj = c->gj;
  a.status = c->status;
  int rc = launch_setup(a, s);
  if (rc) return rc;
  if (c->prm.precision == PC_MIXED) {
    c->f32_ready = false;
    c->tc_ready = false;
    if (c->tc) {
      rc = tc_prepare_operators(c->tc, c->W, c->T, c->cA, 1.0 / c->sO, s);
      if (rc) return rc;
      c->tc_ready = true;
    }
    c->oz_ready = false;
    if (c->oz) {  // the final step's operators: W in SI but for its power of two (the epilogue scales), T_rho / sO
      rc = oz_prepare_operators(c->oz, c->W, c->T, c->sig_scale, 1.0 / c->sO, s);
      if (rc) return rc;
      c->oz_ready = true;
    }
  }
  PC_CUDA_TRY(cudaEventRecord(c->ev_s1, s));
  c->have_design = true;
  c->have_bands = false;
  c->have_grad = false;
  return PC_OK;
}

// ---------------------------------------------------------------------------
template <typename R> struct Ops;
// drop_small: pivot below which a unit-scaled Gram column counts as dependent.
template <> struct Ops<double> {
  typedef double2 C2;
  static constexpr double drop_small = 1e-12;
};
template <> struct Ops<float> {
  typedef float2 C2;
  static constexpr float drop_small = 1e-5f;
};

// A x and Omega x for nvec (selected) vectors with the per-k geometry Q (vector v belongs to k = v / m).
static int apply_fp64(pc_ctx* c, const double2* X, double2* AX, double2* OX, int nvec, int m, const double* Q,
                      double epi, double alpha_omega, double2* E, double2* S, cudaStream_t s, int phase = -1, VecSel sel = {},
                      double alpha_stress = 1.0) {
  const int N = c->N;
  const long long NN = (long long)N * N;
  const double f = 8.0 * (double)N * (double)N;  // algorithmic flops per complex column
  int rc = launch_strain<double>(X, nvec, m, c->geom, Q, E, s, nullptr, sel);
  if (rc) return rc;
  const long long o = (long long)nvec * N;
  const GemmSeg<double> seg[3] = {
      {c->W, E, S, nvec, alpha_stress}, {c->W + NN, E + o, S + o, 5 * nvec, alpha_stress}, {c->T, X, OX, 3 * nvec, alpha_omega, sel}};
  const int slot = phase >= 0 ? ph_begin(c, phase, f * 9.0 * nvec, s) : -1;
  rc = launch_gemms<double>(N, N, N, N, N, seg, 3, s);
  ph_end(c, slot, s);
  if (rc) return rc;
  return launch_epilogue<double>(S, nvec, m, c->geom, Q, epi, epi, AX, s, nullptr, sel);
}

// The same products as apply_fp64 (operators prepared with Omega scaled by 1/sO) from the
// operators' exact 6-bit slices on the tensor cores (oz_gemm.cu): FP64-accurate to about 2e-12
// of the row and column scales.
static int apply_sliced(pc_ctx* c, OzPlan* oz, const double2* X, double2* AX, double2* OX, int nvec, int m,
                        const double* Q, double epi, double2* E, double2* S, cudaStream_t s) {
  const int N = c->N;
  const double f = 8.0 * (double)N * (double)N;  // algorithmic flops per complex column
  int rc = launch_strain<double>(X, nvec, m, c->geom, Q, E, s);
  if (!rc) rc = oz_slice_columns(oz, E, 6 * nvec, 0, s);
  if (!rc) rc = oz_slice_columns(oz, X, 3 * nvec, 6 * nvec, s);
  if (rc) return rc;
  // the three products, one timed launch each: W1 on the dilatation, W2 on the five deviatoric
  // strain components, T_rho / sO on the displacements
  const int which[3] = {0, 1, 2}, col0[3] = {0, 1, 6}, cols[3] = {1, 5, 3};
  double2* out[3] = {S, S + (long long)nvec * N, OX};
  for (int g = 0; g < 3 && !rc; ++g) {
    const int slot = ph_begin(c, PH_RR_GEMM, f * cols[g] * nvec, s);
    rc = oz_gemm(oz, which[g], col0[g] * nvec, cols[g] * nvec, out[g], s);
    ph_end(c, slot, s);
  }
  if (rc) return rc;
  return launch_epilogue<double>(S, nvec, m, c->geom, Q, epi, epi, AX, s);
}

// The FP32 operators of the CUDA-core products: W * (2 pi)^2 V^2 / sA, T_rho / sO and T_f over the former's
// scale are O(1).  Only where the tensor-core plan could not be set up.
static int prepare_f32(pc_ctx* c, cudaStream_t s) {
  if (c->f32_ready) return PC_OK;
  const long long NN = (long long)c->N * c->N;
  int rc = launch_d2f(c->W, c->Wf, 2 * NN, c->cA, s);
  if (!rc) rc = launch_d2f(c->T, c->Tf, NN, 1.0 / c->sO, s);
  if (!rc) rc = launch_d2f(c->T + NN, c->Tf + NN, 2 * NN, 1.0 / c->cA, s);
  c->f32_ready = rc == PC_OK;
  return rc;
}
// The tensor-core plan to use, its operators prepared, or none (and the FP32 operators prepared).
static int ready_f32(pc_ctx* c, TcPlan* plan, bool* tensor, cudaStream_t s) {
  *tensor = plan && tc_available(plan);
  if (!*tensor) return prepare_f32(c, s);
  if (!c->tc_ready) {
    int rc = tc_prepare_operators(c->tc, c->W, c->T, c->cA, 1.0 / c->sO, s);
    if (rc) return rc;
    c->tc_ready = true;
  }
  return PC_OK;
}

// Nondimensional A' X and Omega' X for nvec (selected) FP32 vectors (vector v at k-point k0 + v / m): the
// split-BF16 tensor-core path; the FP32 CUDA-core GEMM only without a tensor-core plan.
static int apply_fp32(pc_ctx* c, const float2* X, float2* AX, float2* OX, int nvec, int m, int k0,
                      cudaStream_t s, TcPlan* plan = nullptr, VecSel sel = {}) {
  const double* Q = c->Q + 3LL * k0;
  const float4* Kf = c->Kf ? c->Kf + (long long)k0 * c->N : nullptr;
  if (!plan) plan = c->tc;
  bool tensor;
  int rc = ready_f32(c, plan, &tensor, s);
  if (rc) return rc;
  if (tensor) return tc_apply(plan, X, AX, OX, nvec, m, c->geom, Q, s, Kf, sel);
  const int N = c->N;
  const long long NN = (long long)N * N;
  float2* E = (float2*)c->E;
  float2* S = (float2*)c->S;
  rc = launch_strain<float>(X, nvec, m, c->geom, Q, E, s, Kf, sel);
  if (rc) return rc;
  const long long o = (long long)nvec * N;
  const GemmSeg<float> seg[3] = {
      {c->Wf, E, S, nvec, 1.f}, {c->Wf + NN, E + o, S + o, 5 * nvec, 1.f}, {c->Tf, X, OX, 3 * nvec, 1.f, sel}};
  rc = launch_gemms<float>(N, N, N, N, N, seg, 3, s);
  if (rc) return rc;
  return launch_epilogue<float>(S, nvec, m, c->geom, Q, 1.0f, 1.0f, AX, s, Kf, sel);
}

// A subset of the k-points run by one host thread on one stream: k in [k0, k0 + nk).
struct KSet {
  int k0 = 0, nk = 0;
  cudaStream_t s = nullptr;
  OpenSet open;             // its k-points still iterated (indices from k0), on the device
  int* h_count = nullptr;   // pinned host copy of open.count
  int unconv = 0, iterations = 0, group = 0;
  unsigned char* rr_scratch = nullptr;  // of its projected problems, rr_slots of them a launch
  int rr_slots = 0;
  TcPlan* tc = nullptr;     // tensor-core workspaces of this subset
  OzPlan* oz = nullptr;     // sliced products of this subset's final Rayleigh-Ritz step (or NULL)
};

static OpenSet open_set(const pc_ctx* c, int k0, int group) {
  return OpenSet{c->open_k + k0, c->open_v + (long long)k0 * c->m, c->fresh_k + k0, c->d_count + 4 * group,
                 c->open_pos + (long long)k0 * c->m};
}

// A X and Omega X of the nsel selected vectors of the subset.
template <typename R>
static int apply_R(pc_ctx* c, const KSet& ks, const typename Ops<R>::C2* X, typename Ops<R>::C2* AX,
                   typename Ops<R>::C2* OX, int nsel, VecSel sel) {
  if constexpr (std::is_same<R, double>::value)
    return apply_fp64(c, X, AX, OX, nsel, c->m, c->Q + 3 * ks.k0, c->cA, 1.0 / c->sO, (double2*)c->E, (double2*)c->S,
                      ks.s, -1, sel);
  else
    return apply_fp32(c, X, AX, OX, nsel, c->m, ks.k0, ks.s, ks.tc, sel);
}
// The preconditioner (waves.cuh) on the ncol unconverged columns of the nopen open k-points.
template <typename R>
static int precond_R(pc_ctx* c, const KSet& ks, const typename Ops<R>::C2* AX, const typename Ops<R>::C2* OX, const R* lam,
                     int nopen, int ncol, double* ref, typename Ops<R>::C2* W, typename Ops<R>::C2* AW,
                     typename Ops<R>::C2* OW) {
  typedef typename Ops<R>::C2 C2;
  const int N = c->N, m = c->m, nb = c->nb;
  const double* Q = c->Q + 3 * ks.k0;
  const float4* Kf = c->Kf ? c->Kf + (long long)ks.k0 * N : nullptr;
  const C2* S = (const C2*)c->S;
  bool tensor = false;
  int rc = PC_OK;
  if constexpr (std::is_same<R, float>::value) {
    TcPlan* plan = ks.tc ? ks.tc : c->tc;
    rc = ready_f32(c, plan, &tensor, ks.s);
    if (!rc && tensor) rc = tc_precond(plan, AX, OX, lam, ks.open.vlist, ncol, m, nb, c->geom, Q, ref, W, &S, ks.s, Kf);
    if (rc) return rc;
  }
  if (!tensor) {
    C2 *E = (C2*)c->E, *So = (C2*)c->S;
    const long long NN = (long long)N * N, o = (long long)ncol * N;
    rc = launch_prec_in<R>(AX, OX, lam, ks.open.vlist, ncol, m, nb, c->geom, Q, ref, W, E, ks.s, Kf);
    if (rc) return rc;
    const C2* T = std::is_same<R, double>::value ? (const C2*)c->T : (const C2*)c->Tf;
    const R al = std::is_same<R, double>::value ? (R)(1.0 / c->cA) : (R)1;
    const GemmSeg<R> seg[2] = {{T + NN, E, So, ncol, al}, {T + 2 * NN, E + o, So + o, 5 * ncol, al}};
    rc = launch_gemms<R>(N, N, N, N, N, seg, 2, ks.s);
    if (rc) return rc;
  }
  return launch_prec_out<R>(S, lam, ks.open.klist, ks.open.vpos, nopen, ncol, m, nb, c->geom, Q, ref, W, AW, OW, ks.s, Kf);
}

template <typename R>
static UpdateArgs<R> upd(pc_ctx* c, int nk, int nblk, int identity_last, MatRef<R> Cmat, int cld, int mout,
                         const int* klist = nullptr) {
  UpdateArgs<R> u = {};
  u.nblk = nblk;
  u.identity_last = identity_last;
  u.C = Cmat;
  u.cld = cld;
  u.klist = klist;
  u.m = c->m;
  u.mout = mout;
  u.n3 = 3 * c->N;
  u.nk = nk;
  u.in_kstride = (long long)c->m * 3 * c->N;
  u.out_kstride = (long long)mout * 3 * c->N;
  u.ntrip = 3;
  u.status = c->status;
  return u;
}
// nk matrices of nel entries, one after the other.
template <typename R>
static MatRef<R> mats(const void* p, long long nel) {
  MatRef<R> r;
  r.p = (const typename cplx_t<R>::type*)p;
  r.nel = nel;
  return r;
}

// k-points of the pc_bands calls running in this process (from other threads too): how many projected problems
// may want an SM at once.  It only chooses between launch forms of the same bits.
static std::atomic<long long> g_running_k{0};
struct RunningK {
  const long long nk;
  explicit RunningK(int n) : nk(n) { g_running_k += nk; }
  ~RunningK() { g_running_k -= nk; }
};

// The projected problems (Rayleigh-Ritz pencil, conjugate-direction coefficients and the
// Cholesky-QR of the search directions) of the mixed form's block iteration take FP32
// Gram matrices; they are solved in FP32 (their inputs carry FP32 accuracy, and an FP64
// solve costs ~60x more on this part's FP64 units).  The final Rayleigh-Ritz step always runs
// in FP64 on FP64 Grams.
template <typename R> struct SmallTol;
template <> struct SmallTol<double> { static constexpr double pdir_abs = 1e-26; };
// FP32: at norms of a few roundings (1e-7) what is left of a direction is rounding, and normalising it puts that into
// P and, ten million times enlarged, into the carried A P and Omega P: of 16 start blocks on uniform SC cells (N = 125, 21
// bands, 40 k-points) eight then broke down at 1e-14, with 41 to 50 iterations and frequencies off by up to 2.4e-6;
// at 1e-12 all take 17 to 19, for 7 % more iterations (and no more time) over a mix of designs.
template <> struct SmallTol<float> { static constexpr float pdir_abs = 1e-12f; };

template <typename R>
static int small_rr_any(pc_ctx* c, const KSet& ks, int nk, const MatRef<R>& GA, const MatRef<R>& GO, int n, int m,
                        const int* klist, R* lam, typename Ops<R>::C2* cX, typename Ops<R>::C2* cP, cudaStream_t s) {
  // the conjugate directions come from the same CTAs
  if constexpr (std::is_same<R, float>::value)
    return launch_small_rr32(GA, GO, n, m, nk, Ops<R>::drop_small, klist, lam, cX, cP, SmallTol<R>::pdir_abs,
                             c->status, c->profiling ? c->small_flops : nullptr, ks.rr_scratch, c->sr_stride, ks.rr_slots, s);
  else
    return launch_small_rr64(GA, GO, n, m, nk, Ops<R>::drop_small, klist, lam, cX, cP, SmallTol<R>::pdir_abs,
                             c->status, ks.rr_scratch, c->sr_stride, ks.rr_slots, g_running_k.load() - c->nk, s);
}
// The batched block iteration (all k at once).  Per iteration and k:
//   R = A X - Omega X Lambda,  W = P R on the unconverged columns (P: waves.cuh);
//   W <- W - X (OX^H W) - P (OP^H W); AW, OW = A W, Omega W (explicit products);
//   W <- W T (Cholesky-QR in the Omega metric, dependent directions dropped);
//   Rayleigh-Ritz on S = [X W P]: X <- S cX, P <- S cP (cP from the small space).
// k-points whose wanted bands are all converged are locked: their block goes to the FP64 step's input
// and every later launch covers the open ones only (klist), the operator products the unconverged columns
// only (vlist).  With tolerance 1e-4 the iterations of a call average 0.8 of the k-points and 0.55 of the
// columns on the design workloads, less at tighter ones.
// Gram and update launches with their algorithmic flops and bytes recorded while profiling.
template <typename R>
static int gram_ph(pc_ctx* c, BlockList<R> A, int na, BlockList<R> B, int nbk, int nk, int m, int n3, R scale,
                   typename cplx_t<R>::type* part, typename cplx_t<R>::type* G, MatRef<R>* out, const int* klist,
                   int max_split, cudaStream_t s) {
  const double esz = sizeof(typename cplx_t<R>::type);
  const double fl = 8.0 * n3 * (double)(na * m) * (double)(nbk * m) * nk;
  const double by = esz * ((double)(na + nbk) * m * n3 + (double)(na * m) * (nbk * m)) * nk;
  int sl = ph_begin(c, PH_GRAM, fl, s, by);
  int rc = launch_gram<R>(A, na, B, nbk, nk, m, n3, scale, part, G, out, s, c->status, klist, max_split);
  ph_end(c, sl, s);
  return rc;
}
template <typename R>
static int update_ph(pc_ctx* c, const UpdateArgs<R>& u, cudaStream_t s) {
  const double esz = sizeof(typename cplx_t<R>::type);
  const int nsum = u.identity_last ? u.nblk - 1 : u.nblk;
  const int nset = u.C2nd.p ? 2 : 1;
  const double fl = 8.0 * u.n3 * (double)(nsum * u.m) * u.mout * nset * u.nk * u.ntrip;
  const double by = esz * ((double)u.nblk * u.m + (double)nset * u.mout) * u.n3 * (double)u.nk * u.ntrip;
  int sl = ph_begin(c, PH_UPDATE, fl, s, by);
  int rc = launch_update<R>(u, s);
  ph_end(c, sl, s);
  return rc;
}

template <typename R>
static int run_block_iteration(pc_ctx* c, KSet& ks) {
  typedef typename Ops<R>::C2 C2;
  const int m = c->m, nk = ks.nk, n3 = 3 * c->N, nb = c->nb, k0 = ks.k0;
  cudaStream_t s = ks.s;
  // per-k buffers of this subset (the small workspaces at their largest per-k size)
  const long long G1 = 72LL * 72;
  C2* b[15];
  for (int i = 0; i < 15; ++i) b[i] = (C2*)c->blk[i] + (long long)k0 * m * n3;
  const double* Qk = c->Q + 3 * k0;
  int* kdone = c->kdone + k0;
  int* active = c->active + (long long)k0 * m;
  double* rnorm = c->rnorm + (long long)k0 * m;
  double* sbest = c->stall_best + k0;
  int* ssince = c->stall_since + k0;
  C2 *X = b[0], *AX = b[1], *OX = b[2], *Wb = b[3], *AW = b[4], *OW = b[5], *P = b[6], *AP = b[7], *OP = b[8];
  C2 *Xn = b[9], *AXn = b[10], *OXn = b[11], *Pn = b[12], *APn = b[13], *OPn = b[14];
  // Partial Gram matrices: room for 8 of the largest per k-point of the subset.  The FP32 consumers add
  // them up themselves, so that two products are held at once; the FP64 ones are reduced by a launch.
  const bool two = std::is_same<R, float>::value;
  const long long room = (two ? 4 : 8) * G1 * nk;  // entries per product
  C2 *part = (C2*)c->gpart + k0 * 8 * G1, *part2 = two ? part + room : part;
  auto splits = [&](int nopen, int nel) { return (int)std::min<long long>(8, room / ((long long)nopen * nel)); };
  C2 *GA = (C2*)c->GA + k0 * G1, *GO = (C2*)c->GO + k0 * G1, *Cc = (C2*)c->Cc + k0 * G1, *Ct = (C2*)c->Ct + k0 * G1;
  R* lam = (R*)c->lam + (long long)k0 * m;
  double2* Xd = c->Xd + (long long)k0 * m * n3;  // the final blocks
  int rc;
#define TRY(x) do { rc = (x); if (rc) return rc; } while (0)
  const OpenSet& o = ks.open;
  const int* klist = o.klist;
  int nopen = nk;
  MatRef<R> gA, gO;  // the Gram products at hand
  PC_CUDA_TRY(cudaMemsetAsync(kdone, 0, sizeof(int) * nk, s));
  PC_CUDA_TRY(cudaMemsetAsync(sbest, 0, sizeof(double) * nk, s));
  PC_CUDA_TRY(cudaMemsetAsync(ssince, 0, sizeof(int) * nk, s));
  if (c->import_pending || (c->warm && c->warm_ready)) {
    // warm start: the final Ritz block of the last pc_bands (or the imported one), FP64 in Th
    const double2* th = c->Th + (long long)k0 * m * n3;
    const long long cnt = (long long)nk * m * n3;
    if constexpr (std::is_same<R, float>::value) {
      TRY(launch_d2f(th, (float2*)X, cnt, 1.0, s));
    } else {
      PC_CUDA_TRY(cudaMemcpyAsync(X, th, sizeof(double2) * cnt, cudaMemcpyDeviceToDevice, s));
    }
  } else {
    TRY(launch_init_guess<R>(X, nk, m, c->geom, Qk, c->seed, s));
  }
  double* ref = c->prec_ref + 3 * ks.group;
  TRY(launch_open_all(o, nk, c->pr, c->chi_mean, ref, s));
  TRY(apply_R<R>(c, ks, X, AX, OX, nk * m, VecSel{}));
  {
    BlockList<R> A1 = {{X, nullptr, nullptr}}, B1 = {{AX, nullptr, nullptr}}, B2 = {{OX, nullptr, nullptr}};
    const int sp = splits(nk, m * m);
    TRY(gram_ph<R>(c, A1, 1, B1, 1, nk, m, n3, (R)1, part, GA, &gA, klist, sp, s));
    TRY(gram_ph<R>(c, A1, 1, B2, 1, nk, m, n3, (R)1, part2, GO, &gO, klist, sp, s));
    TRY(small_rr_any<R>(c, ks, nk, gA, gO, m, m, klist, lam, Cc, nullptr, s));
    UpdateArgs<R> u = upd<R>(c, nk, 1, 0, mats<R>(Cc, (long long)m * m), m, m, klist);
    u.in[0][0] = X; u.in[1][0] = AX; u.in[2][0] = OX;
    u.out[0] = Xn; u.out[1] = AXn; u.out[2] = OXn;
    TRY(update_ph<R>(c, u, s));
    std::swap(X, Xn); std::swap(AX, AXn); std::swap(OX, OXn);
  }
  bool hasP = false;
  int it = 0;
  ks.unconv = nk;
  for (it = 0; it < c->prm.max_iter; ++it) {
    // The products A X and Omega X are carried along by the same linear combinations as X;
    // their rounding drifts away from the true products.  Every c->refresh iterations they
    // are recomputed from X and the conjugate block is restarted.
    if (it > 0 && it % c->refresh == 0) {
      int sl = ph_begin(c, PH_ITER_APPLY, 8.0 * c->N * (double)c->N * 9.0 * nopen * m, s);
      TRY(apply_R<R>(c, ks, X, AX, OX, nopen * m, VecSel{klist, m}));
      ph_end(c, sl, s);
      hasP = false;
    }
    TRY(launch_resnorm<R>(AX, OX, lam, nk, m, nb, n3, c->prm.tol, rnorm, active, kdone, o, nopen, s, sbest, ssince));
    PC_CUDA_TRY(cudaMemcpyAsync(ks.h_count, o.count, 4 * sizeof(int), cudaMemcpyDeviceToHost, s));
    // While profiling, the stream's idle gap while the host waits for the count and enqueues the
    // next step: from the completion of the copy to the next work the host enqueues.
    const int idle_slot = ph_begin(c, PH_IDLE, 0.0, s);
    PC_CUDA_TRY(cudaStreamSynchronize(s));
    nopen = ks.h_count[0];
    ks.unconv = ks.h_count[3];  // what the call reports: open k-points may have met the tolerance already
    const int ncol = ks.h_count[1], nfresh = ks.h_count[2];
    if (c->debug) {
      const int nv = nk * m;
      std::vector<double> h(nv);
      cudaMemcpy(h.data(), rnorm, sizeof(double) * nv, cudaMemcpyDeviceToHost);
      std::vector<int> kd(nk);
      cudaMemcpy(kd.data(), kdone, sizeof(int) * nk, cudaMemcpyDeviceToHost);
      double mx = 0, mxo = 0;
      int kmx = 0, kmxo = -1;
      for (int k = 0; k < nk; ++k)
        for (int j = 0; j < nb; ++j) {
          if (h[k * m + j] > mx) { mx = h[k * m + j]; kmx = k; }
          if (kd[k] != 1 && h[k * m + j] > mxo) { mxo = h[k * m + j]; kmxo = k; }
        }
      fprintf(stderr, "[pc] k %d+ it %d unconverged_k %d max_res %.3e at k %d; open k: max_res %.3e at k %d\n", k0,
              it, ks.unconv, mx, kmx + k0, mxo, kmxo < 0 ? -1 : kmxo + k0);
      const char* dk = getenv("PC_DEBUG_K");
      if (dk && atoi(dk) >= k0 && atoi(dk) < k0 + nk) {
        int kk = atoi(dk) - k0;
        fprintf(stderr, "[pc]   k %d col res:", kk);
        for (int j = 0; j < m; ++j) fprintf(stderr, " %.1e", h[kk * m + j]);
        fprintf(stderr, "\n");
      }
    }
    ph_end(c, idle_slot, s);
    TRY(launch_store<R>(X, Xd, o.fresh, nfresh, (long long)m * n3, s));
    if (nopen == 0) break;
    {
      int sl = ph_begin(c, PH_ITER_APPLY, 8.0 * c->N * (double)c->N * 6.0 * ncol, s);
      TRY(precond_R<R>(c, ks, AX, OX, lam, nopen, ncol, ref, Wb, AW, OW));
      ph_end(c, sl, s);
    }
    // W <- W - X (OX^H W) - P (OP^H W), before the operator is applied
    {
      const int nproj = hasP ? 2 : 1;
      BlockList<R> A1 = {{OX, OP, nullptr}}, B1 = {{Wb, nullptr, nullptr}};
      TRY(gram_ph<R>(c, A1, nproj, B1, 1, nopen, m, n3, (R)-1, part, Ct, &gO, klist, splits(nopen, nproj * m * m), s));
      UpdateArgs<R> u = upd<R>(c, nopen, nproj + 1, 1, gO, m, m, klist);
      u.ntrip = 1;
      u.in[0][0] = X;
      if (hasP) { u.in[0][1] = P; u.in[0][2] = Wb; } else { u.in[0][1] = Wb; }
      u.out[0] = Wb;
      TRY(update_ph<R>(c, u, s));
    }
    {
      int sl = ph_begin(c, PH_ITER_APPLY, 8.0 * c->N * (double)c->N * 9.0 * ncol, s);
      TRY(apply_R<R>(c, ks, Wb, AW, OW, ncol, VecSel{o.vlist, 1}));
      ph_end(c, sl, s);
    }
    // W <- W T with T^H (W^H Omega W) T = I, dependent directions dropped
    {
      BlockList<R> A1 = {{Wb, nullptr, nullptr}}, B1 = {{OW, nullptr, nullptr}};
      TRY(gram_ph<R>(c, A1, 1, B1, 1, nopen, m, n3, (R)1, part, GO, &gO, klist, splits(nopen, m * m), s));
      int sl = ph_begin(c, PH_SMALL, 0.0, s);
      TRY(launch_small_chol<R>(gO, m, nopen, Ops<R>::drop_small, Cc, s));
      ph_end(c, sl, s);
      UpdateArgs<R> u = upd<R>(c, nopen, 1, 0, mats<R>(Cc, (long long)m * m), m, m, klist);
      u.in[0][0] = Wb; u.in[1][0] = AW; u.in[2][0] = OW;
      u.out[0] = Wb; u.out[1] = AW; u.out[2] = OW;
      TRY(update_ph<R>(c, u, s));
    }
    // Rayleigh-Ritz on S = [X W P]
    const int ns = hasP ? 3 : 2;
    const int n = ns * m;
    BlockList<R> S1 = {{X, Wb, P}}, SA = {{AX, AW, AP}}, SO = {{OX, OW, OP}};
    const int sp = splits(nopen, n * n);
    TRY(gram_ph<R>(c, S1, ns, SA, ns, nopen, m, n3, (R)1, part, GA, &gA, klist, sp, s));
    TRY(gram_ph<R>(c, S1, ns, SO, ns, nopen, m, n3, (R)1, part2, GO, &gO, klist, sp, s));
    {
      int sl = ph_begin(c, PH_SMALL, 0.0, s);
      TRY(small_rr_any<R>(c, ks, nopen, gA, gO, n, m, klist, lam, Cc, Ct, s));
      ph_end(c, sl, s);
    }
    {
      UpdateArgs<R> u = upd<R>(c, nopen, ns, 0, mats<R>(Cc, (long long)n * m), m, m, klist);
      u.in[0][0] = X; u.in[0][1] = Wb; u.in[0][2] = P;
      u.in[1][0] = AX; u.in[1][1] = AW; u.in[1][2] = AP;
      u.in[2][0] = OX; u.in[2][1] = OW; u.in[2][2] = OP;
      u.out[0] = Xn; u.out[1] = AXn; u.out[2] = OXn;
      u.C2nd = mats<R>(Ct, (long long)n * m);  // conjugate directions from the same inputs
      u.out2[0] = Pn; u.out2[1] = APn; u.out2[2] = OPn;
      TRY(update_ph<R>(c, u, s));
    }
    std::swap(X, Xn); std::swap(AX, AXn); std::swap(OX, OXn);
    std::swap(P, Pn); std::swap(AP, APn); std::swap(OP, OPn);
    hasP = true;
  }
  ks.iterations = it;
  // out of iterations: the blocks still open are what they are
  if (nopen > 0) TRY(launch_store<R>(X, Xd, klist, nopen, (long long)m * n3, s));
#undef TRY
  return PC_OK;
}

static int fp64_rayleigh_ritz(pc_ctx* c, const KSet& ks);

// The mixed form's block iteration on groups of the k-points, each on its own non-blocking
// stream and host thread.  The groups are independent problems; running them concurrently
// lets the latency-bound projected problems of one group overlap the bandwidth- and
// tensor-bound products of the others.  Forked from and joined back to the caller's stream
// with events.
static int run_split_iteration(pc_ctx* c, cudaStream_t s) {
  if (!c->tc_ready) {
    int rc = tc_prepare_operators(c->tc, c->W, c->T, c->cA, 1.0 / c->sO, s);
    if (rc) return rc;
    c->tc_ready = true;
  }
  const int ng = kgroups(c, c->nk);
  PC_CUDA_TRY(cudaEventRecord(c->ev_fork, s));
  KSet ks[kMaxGroups];
  for (int g = 0; g < ng; ++g) {
    ks[g].k0 = (int)(((long long)c->nk * g) / ng);
    ks[g].nk = (int)(((long long)c->nk * (g + 1)) / ng) - ks[g].k0;
    ks[g].s = c->sk[g];
    ks[g].group = g;
    ks[g].open = open_set(c, ks[g].k0, g);
    ks[g].h_count = c->h_count + 4 * g;
    ks[g].rr_scratch = c->sr_scratch + rr_first(c->nk, ng, g) * c->sr_stride;
    ks[g].rr_slots = rr_problems_per_launch(ks[g].nk, device_sms());
    ks[g].tc = g ? c->tcg[g] : c->tc;
    ks[g].oz = (c->oz_ready && c->oz) ? (g ? c->ozg[g] : c->oz) : nullptr;
    PC_CUDA_TRY(cudaStreamWaitEvent(c->sk[g], c->ev_fork, 0));
  }
  int rcs[kMaxGroups] = {}, dev = 0;
  PC_CUDA_TRY(cudaGetDevice(&dev));
  std::vector<std::thread> others;
  for (int g = 1; g < ng; ++g)
    others.emplace_back([&, g] {
      // a new host thread starts on device 0: adopt the caller's device first
      if (cudaSetDevice(dev) != cudaSuccess) { rcs[g] = PC_ECUDA; return; }
      rcs[g] = run_block_iteration<float>(c, ks[g]);
      if (!rcs[g]) rcs[g] = fp64_rayleigh_ritz(c, ks[g]);
    });
  rcs[0] = run_block_iteration<float>(c, ks[0]);
  if (!rcs[0]) rcs[0] = fp64_rayleigh_ritz(c, ks[0]);
  for (auto& t : others) t.join();
  c->iterations = 0;
  c->unconv = 0;
  int rc = PC_OK;
  for (int g = 0; g < ng; ++g) {
    PC_CUDA_TRY(cudaEventRecord(c->ev_join[g], c->sk[g]));
    PC_CUDA_TRY(cudaStreamWaitEvent(s, c->ev_join[g], 0));
    c->iterations = std::max(c->iterations, ks[g].iterations);
    c->unconv += ks[g].unconv;
    if (!rc) rc = rcs[g];
  }
  return rc;
}

// One FP64 Rayleigh-Ritz step on the final block: FP64 operator, FP64 Gram matrices,
// FP64 projected eigenproblem; yields lambda, theta and the stresses of theta.
static int fp64_rayleigh_ritz(pc_ctx* c, const KSet& ks) {
  const int m = c->m, nk = ks.nk, N = c->N, n3 = 3 * N, k0 = ks.k0;
  cudaStream_t s = ks.s;
  const long long nvec = (long long)nk * m, nvec_all = (long long)c->nk * m;
  const long long vo = (long long)k0 * m;  // first vector of this subset
  // this subset's FP64 workspaces: vectors at their global offset; strain/stress stacks
  // [6][nvec][N] compact inside the subset's share of Ed/Sd
  double2* AXd = c->AXd + vo * n3;
  double2* OXd = c->OXd + vo * n3;
  double2* Ed = c->Ed + 6 * vo * N;
  double2* Sd = c->Sd + 6 * vo * N;
  double2* GAd = c->GAd + (long long)k0 * m * m;
  double2* GOd = c->GOd + (long long)k0 * m * m;
  double2* Cd = c->Cd + (long long)k0 * m * m;
  double2* gpartd = c->gpartd + 8LL * k0 * m * m;
  double* lamd = c->lamd + vo;
  int rc;
  const double2* X = c->Xd + vo * n3;
  const double epi = c->cA / c->sig_scale;
  if (ks.oz)
    rc = apply_sliced(c, ks.oz, X, AXd, OXd, (int)nvec, m, c->Q + 3 * k0, epi, Ed, Sd, s);
  else
    rc = apply_fp64(c, X, AXd, OXd, (int)nvec, m, c->Q + 3 * k0, epi, 1.0 / c->sO, Ed, Sd, s, PH_RR_GEMM, {}, c->sig_scale);
  if (rc) return rc;
  BlockList<double> A1 = {{X, nullptr, nullptr}}, B1 = {{AXd, nullptr, nullptr}}, B2 = {{OXd, nullptr, nullptr}};
  MatRef<double> gA, gO;
  rc = launch_gram<double>(A1, 1, B1, 1, nk, m, n3, 1.0, gpartd, GAd, &gA, s);
  if (rc) return rc;
  rc = launch_gram<double>(A1, 1, B2, 1, nk, m, n3, 1.0, gpartd, GOd, &gO, s);
  if (rc) return rc;
  rc = launch_small_rr64(gA, gO, m, m, nk, 1e-12, nullptr, lamd, Cd, nullptr, 0.0, c->status,
                         ks.rr_scratch, c->sr_stride, ks.rr_slots, 0, s);
  if (rc) return rc;
  // theta = X C; A theta and Omega theta for the residual report
  UpdateArgs<double> u = upd<double>(c, nk, 1, 0, mats<double>(Cd, (long long)m * m), m, m);
  u.in[0][0] = X; u.in[1][0] = AXd; u.in[2][0] = OXd;
  // the strain stacks (6 nvec N = 2 nvec 3N entries) are free after the apply: they take
  // A theta and Omega theta for the residual report
  double2* Ath = Ed;
  double2* Oth = Ed + nvec * n3;
  u.out[0] = c->Th + vo * n3;
  u.out[1] = Ath;
  u.out[2] = Oth;
  rc = launch_update<double>(u, s);
  if (rc) return rc;
  PC_CUDA_TRY(cudaMemsetAsync(c->kdone_f + k0, 0, sizeof(int) * nk, s));
  rc = launch_resnorm<double>(Ath, Oth, lamd, nk, m, c->nb, n3, c->prm.tol, c->rnormd + vo, c->actived + vo,
                              c->kdone_f + k0, OpenSet{nullptr, nullptr, nullptr, ks.open.count, nullptr}, nk, s);
  if (rc) return rc;
  // stresses of theta in the global layout [6][nk m][N]: St[s] = Sd[s] C
  for (int half = 0; half < 2; ++half) {
    UpdateArgs<double> v = upd<double>(c, nk, 1, 0, mats<double>(Cd, (long long)m * m), m, m);
    v.n3 = N;
    v.in_kstride = (long long)m * N;
    v.out_kstride = (long long)m * N;
    for (int t = 0; t < 3; ++t) {
      int sidx = half * 3 + t;
      v.in[t][0] = Sd + (long long)sidx * nvec * N;
      v.out[t] = c->St + (long long)sidx * nvec_all * N + vo * N;
    }
    rc = launch_update<double>(v, s);
    if (rc) return rc;
  }
  return PC_OK;
}

extern "C" int pc_bands(pc_ctx* c, double* omega, void* stream) {
  if (!c || !omega) return PC_EINVAL;
  cudaGetLastError();  // launch checks below report only this call's launches
  if (!c->have_design || c->nk == 0) return PC_ESTATE;
  const RunningK running(c->nk);
  cudaStream_t s = (cudaStream_t)stream;
  PC_CUDA_TRY(cudaEventRecord(c->ev0, s));
  int sl = ph_begin(c, PH_LOOP, 0.0, s);
  int rc;
  bool split = c->split && c->prm.precision == PC_MIXED && c->tc &&
               tc_available(c->tc) && kgroups(c, c->nk) >= 2;
  for (int g = 1; split && g < kgroups(c, c->nk); ++g) split = c->tcg[g] && tc_available(c->tcg[g]);
  if (split) {
    // each k group runs its FP64 Rayleigh-Ritz step as soon as its own iteration ends
    rc = run_split_iteration(c, s);
    ph_end(c, sl, s);
    if (rc) return rc;
  } else {
    KSet ks;
    ks.k0 = 0;
    ks.nk = c->nk;
    ks.s = s;
    ks.open = open_set(c, 0, 0);
    ks.h_count = c->h_count;
    ks.rr_scratch = c->sr_scratch;
    ks.rr_slots = rr_problems_per_launch(c->nk, device_sms());
    ks.tc = c->tc;
    ks.oz = (c->oz_ready && c->oz) ? c->oz : nullptr;
    rc = (c->prm.precision == PC_FP64) ? run_block_iteration<double>(c, ks) : run_block_iteration<float>(c, ks);
    c->iterations = ks.iterations;
    c->unconv = ks.unconv;
    ph_end(c, sl, s);
    if (rc) return rc;
    sl = ph_begin(c, PH_FINAL, 0.0, s);
    rc = fp64_rayleigh_ritz(c, ks);
    ph_end(c, sl, s);
    if (rc) return rc;
  }
  rc = launch_omega(c->lamd, c->nk, c->nb, c->m, c->lref, omega, c->lam_nd, s);
  if (rc) return rc;
  PC_CUDA_TRY(cudaEventRecord(c->ev1, s));
  c->have_bands = true;
  c->warm_ready = true;
  c->import_pending = false;
  c->have_grad = false;
  return PC_OK;
}

// Objective weights (exact, smooth or user-given) and the adjoint gradient they select.
static int gap_and_grad_impl(pc_ctx* c, int n_lower, int mode, double beta, const double* w, double* gap,
                             double* grad, void* stream) {
  if (!c->have_bands) return PC_ESTATE;
  // Refused before anything is enqueued: the adjoint's shared staging must fit.
  if (grad && adjoint_staging_bytes(c->prm.M, c->prm.n[1], c->prm.n[2], c->prm.precision == PC_MIXED) >
                  kAdjointStagingMax)
    return PC_EINVAL;
  cudaGetLastError();  // launch checks below report only this call's launches
  cudaStream_t s = (cudaStream_t)stream;
  PC_CUDA_TRY(cudaEventRecord(c->ev_g0, s));
  GapArgs g;
  g.lam = c->lam_nd;
  g.nk = c->nk; g.nb = c->nb; g.n_lower = n_lower; g.mode = mode;
  g.lref = c->lref;
  g.rel_tol = c->prm.precision == PC_MIXED ? PC_CLUSTER_TOL_MIXED : PC_CLUSTER_TOL_FP64;
  g.ks_beta = beta;
  g.w_user = w;
  g.gap_out = gap;
  g.weights = c->weights;
  g.pairs = c->pairs;
  g.npairs = c->npairs;
  int rc = launch_gap(g, s);
  if (rc) return rc;
  if (grad) {
    AdjointArgs a;
    a.theta = c->Th;
    a.sig = c->St;
    a.lam = c->lam_nd;
    a.weights = c->weights;
    a.pairs = c->pairs;
    a.npairs = c->npairs;
    a.max_pairs = c->nk * c->nb;
    a.nk = c->nk; a.nb = c->nb; a.m = c->m; a.N = c->N; a.M = c->prm.M;
    a.n0 = c->prm.n[0]; a.n1 = c->prm.n[1]; a.n2 = c->prm.n[2];
    a.lref = c->lref;
    a.inv_sO = 1.0 / c->sO;
    a.d_rho = c->mc.rho1 - c->mc.rho0;
    a.dfc = c->dfc;
    a.w_scale = c->w_scale;
    a.w_inv = 1.0 / c->w_scale;
    const double tv = 2.0 * M_PI * c->V / c->sig_scale;
    a.two_pi_V_sq = tv * tv;
    a.ve = c->ve;
    a.dchi = c->dchi;
    a.t2 = c->adj_t2;
    a.phases = c->adj_ph;
    a.part = c->adj_part;
    a.grad = grad;
    int sl = ph_begin(c, PH_GRAD, 0.0, s);
    rc = launch_adjoint(a, c->prm.precision == PC_MIXED, s);
    ph_end(c, sl, s);
    if (rc) return rc;
  }
  PC_CUDA_TRY(cudaEventRecord(c->ev_g1, s));
  c->have_grad_events = true;
  c->have_grad = true;
  return PC_OK;
}

extern "C" int pc_gap_and_grad(pc_ctx* c, int n_lower, int mode, const double* w, double* gap, double* grad,
                               void* stream) {
  if (!c || !gap) return PC_EINVAL;
  if (mode != PC_GAP_OMEGA && mode != PC_GAP_LAMBDA && mode != PC_GRAD_ALLBANDS) return PC_EINVAL;
  if (mode == PC_GRAD_ALLBANDS && !w) return PC_EINVAL;
  if (mode != PC_GRAD_ALLBANDS && (n_lower < 1 || n_lower >= c->nb)) return PC_EINVAL;
  return gap_and_grad_impl(c, n_lower, mode, 0.0, w, gap, grad, stream);
}

extern "C" int pc_gap_ks_and_grad(pc_ctx* c, int n_lower, double beta, double* gap, double* grad, void* stream) {
  if (!c || !gap) return PC_EINVAL;
  if (n_lower < 1 || n_lower >= c->nb || !(beta > 0.0) || !(beta < 1e12)) return PC_EINVAL;
  return gap_and_grad_impl(c, n_lower, PC_GAP_KS_INTERNAL, beta, nullptr, gap, grad, stream);
}

extern "C" int pc_get_stats(pc_ctx* c, pc_stats* out) {
  if (!c || !out) return PC_EINVAL;
  PC_CUDA_TRY(cudaDeviceSynchronize());
  memset(out, 0, sizeof(*out));
  int st = 0;
  PC_CUDA_TRY(cudaMemcpy(&st, c->status, sizeof(int), cudaMemcpyDeviceToHost));
  out->iterations = c->iterations;
  out->unconverged_k = c->unconv;
  out->nk = c->nk;
  out->N = c->N;
  out->block = c->m;
  if (c->have_bands && c->nk > 0) {
    const int nvec = c->nk * c->m;
    double* h = (double*)malloc(sizeof(double) * nvec);
    if (h) {
      cudaMemcpy(h, c->rnormd, sizeof(double) * nvec, cudaMemcpyDeviceToHost);
      double mx = 0;
      for (int k = 0; k < c->nk; ++k)
        for (int j = 0; j < c->nb; ++j) mx = std::max(mx, h[k * c->m + j]);
      out->max_residual = mx;
      free(h);
    }
  }
  if (st == PC_OK && c->unconv > 0) st = PC_ENOCONV;
  float ms = 0;
  if (c->have_design && cudaEventElapsedTime(&ms, c->ev_s0, c->ev_s1) == cudaSuccess) out->ms_setup = ms;
  if (c->have_bands && cudaEventElapsedTime(&ms, c->ev0, c->ev1) == cudaSuccess) out->ms_bands = ms;
  if (c->have_grad_events && cudaEventElapsedTime(&ms, c->ev_g0, c->ev_g1) == cudaSuccess) out->ms_grad = ms;
  cudaGetLastError();  // a query on events of an unfinished call must not leak into later launch checks
  out->launches = g_pc_launches - c->launch_base;
  ph_collect(c);
  out->ms_rr_gemm = c->ph_ms[PH_RR_GEMM];
  out->rr_gemm_launches = c->ph_count[PH_RR_GEMM];
  out->rr_gemm_flops = c->ph_flops[PH_RR_GEMM];
  out->rr_sliced = (c->oz_ready && c->oz) ? 1 : 0;
  out->ms_iter_apply = c->ph_ms[PH_ITER_APPLY];
  out->iter_apply_calls = c->ph_count[PH_ITER_APPLY];
  out->iter_apply_flops = c->ph_flops[PH_ITER_APPLY];
  out->ms_small = c->ph_ms[PH_SMALL];
  out->small_calls = c->ph_count[PH_SMALL];
  out->ms_grad_kernels = c->ph_ms[PH_GRAD];
  out->ms_gram = c->ph_ms[PH_GRAM];
  out->gram_launches = c->ph_count[PH_GRAM];
  out->gram_flops = c->ph_flops[PH_GRAM];
  out->gram_bytes = c->ph_bytes[PH_GRAM];
  out->ms_update = c->ph_ms[PH_UPDATE];
  out->update_launches = c->ph_count[PH_UPDATE];
  out->update_flops = c->ph_flops[PH_UPDATE];
  out->update_bytes = c->ph_bytes[PH_UPDATE];
  out->ms_iteration_loop = c->ph_ms[PH_LOOP];
  PC_CUDA_TRY(cudaMemcpy(&out->small_flops, c->small_flops, sizeof(double), cudaMemcpyDeviceToHost));
  out->grad_flops_per_pair = c->grad_flops_per_pair;
  if (c->have_grad && c->npairs) {
    int np = 0;
    PC_CUDA_TRY(cudaMemcpy(&np, c->npairs, sizeof(int), cudaMemcpyDeviceToHost));
    out->grad_pairs = np;
  }
  out->ms_final_rr = c->ph_ms[PH_FINAL];
  out->ms_host_idle = c->ph_ms[PH_IDLE];
  out->status = st;
  return st;
}

extern "C" int pc_clear_status(pc_ctx* c) {
  if (!c) return PC_EINVAL;
  PC_CUDA_TRY(cudaMemset(c->status, 0, sizeof(int)));
  c->launch_base = g_pc_launches;
  return PC_OK;
}

extern "C" int pc_set_profiling(pc_ctx* c, int on) {
  if (!c) return PC_EINVAL;
  PC_CUDA_TRY(cudaDeviceSynchronize());
  ph_collect(c);
  for (int i = 0; i < PH_COUNT; ++i) { c->ph_ms[i] = 0; c->ph_flops[i] = 0; c->ph_bytes[i] = 0; c->ph_count[i] = 0; }
  PC_CUDA_TRY(cudaMemset(c->small_flops, 0, sizeof(double)));
  c->profiling = on ? 1 : 0;
  return PC_OK;
}

// FMA throughput probe: every thread runs 8 independent FMA chains.
template <typename T>
__global__ void k_fma_probe(T* out, int iters, T a, T b) {
  T x[8];
  for (int i = 0; i < 8; ++i) x[i] = (T)(threadIdx.x + i);
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = x[i] * a + b;
  }
  T s = 0;
  for (int i = 0; i < 8; ++i) s += x[i];
  if (s == (T)-1.2345) out[blockIdx.x] = s;  // keeps the chains alive
}

extern "C" int pc_probe(int what, double* gflops) {
  if (!gflops || (what != 0 && what != 1)) return PC_EINVAL;
  int dev = 0, sms = 0;
  PC_CUDA_TRY(cudaGetDevice(&dev));
  PC_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  void* out = nullptr;
  PC_CUDA_TRY(cudaMalloc(&out, 8 * 65536));
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  const int blocks = sms * 8, threads = 256;
  const int iters = (what == 0) ? 2048 : 65536;
  double best = 0;
  for (int rep = 0; rep < 4; ++rep) {
    cudaEventRecord(e0);
    if (what == 0) k_fma_probe<double><<<blocks, threads>>>((double*)out, iters, 0.999999, 1e-7);
    else k_fma_probe<float><<<blocks, threads>>>((float*)out, iters, 0.999999f, 1e-7f);
    cudaEventRecord(e1);
    if (cudaEventSynchronize(e1) != cudaSuccess) { cudaFree(out); return PC_ECUDA; }
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    double fl = 2.0 * 8.0 * (double)iters * blocks * threads;
    if (rep > 0) best = std::max(best, fl / (ms * 1e-3) / 1e9);
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(out);
  *gflops = best;
  return PC_OK;
}

extern "C" int pc_export(pc_ctx* c, int which, double* host, long long cap, long long* count) {
  if (!c || !count) return PC_EINVAL;
  const long long N = c->N, NN = N * N, L = c->L;
  const void* src = nullptr;
  long long n = 0;
  switch (which) {
    case PC_EXPORT_SFAC: if (!c->have_design) return PC_ESTATE; src = c->sfac; n = 3 * L * L * L * 2; break;
    case PC_EXPORT_TOEP: if (!c->have_design) return PC_ESTATE; src = c->T; n = 3 * NN * 2; break;
    case PC_EXPORT_WINV: if (!c->have_design) return PC_ESTATE; src = c->W; n = 2 * NN * 2; break;
    case PC_EXPORT_LAMBDA: if (!c->have_bands) return PC_ESTATE; n = (long long)c->nk * c->nb; break;
    case PC_EXPORT_EIGVEC: if (!c->have_bands) return PC_ESTATE; n = (long long)c->nk * c->nb * 3 * N * 2; break;
    case PC_EXPORT_WEIGHT: if (!c->have_grad) return PC_ESTATE; src = c->weights; n = (long long)c->nk * c->nb; break;
    case PC_EXPORT_BLOCK: if (!c->warm_ready) return PC_ESTATE; src = c->Th; n = (long long)c->nk * c->m * 3 * N * 2; break;
    default: return PC_EINVAL;
  }
  *count = n;
  if (!host || cap < n) return PC_OK;
  PC_CUDA_TRY(cudaDeviceSynchronize());
  if (which == PC_EXPORT_LAMBDA) {
    PC_CUDA_TRY(cudaMemcpy(host, c->lam_nd, sizeof(double) * n, cudaMemcpyDeviceToHost));
    for (long long i = 0; i < n; ++i) host[i] *= c->lref;
    return PC_OK;
  }
  if (which == PC_EXPORT_EIGVEC) {
    const long long per = 3 * N * 2;
    const double sc = 1.0 / std::sqrt(c->sO);
    for (int k = 0; k < c->nk; ++k) {
      PC_CUDA_TRY(cudaMemcpy(host + (long long)k * c->nb * per, c->Th + (long long)k * c->m * 3 * N,
                             sizeof(double) * per * c->nb, cudaMemcpyDeviceToHost));
    }
    for (long long i = 0; i < n; ++i) host[i] *= sc;
    return PC_OK;
  }
  PC_CUDA_TRY(cudaMemcpy(host, src, sizeof(double) * n, cudaMemcpyDeviceToHost));
  return PC_OK;
}

// Concurrent k groups of the mixed form for the next pc_set_kpoints (batch contexts; 1: one
// stream).  Not exported.
int pc_internal_set_groups(pc_ctx* c, int groups) {
  if (!c || groups < 1 || groups > kMaxGroups) return PC_EINVAL;
  c->groups = groups;
  return PC_OK;
}

extern "C" int pc_set_warm_start(pc_ctx* c, int on) {
  if (!c) return PC_EINVAL;
  c->warm = on ? 1 : 0;
  return PC_OK;
}

extern "C" int pc_import_block(pc_ctx* c, const double* host, long long count) {
  if (!c || !host) return PC_EINVAL;
  if (c->nk == 0) return PC_ESTATE;
  if (count != (long long)c->nk * c->m * 3 * c->N) return PC_EINVAL;
  PC_CUDA_TRY(cudaDeviceSynchronize());
  PC_CUDA_TRY(cudaMemcpy(c->Th, host, sizeof(double2) * count, cudaMemcpyHostToDevice));
  c->import_pending = true;
  return PC_OK;
}

extern "C" int pc_apply_operator(pc_ctx* c, int k, int ncols, const double* x, double* ax, double* ox, void* stream) {
  if (!c || !x || !ax || !ox || ncols < 1) return PC_EINVAL;
  cudaGetLastError();  // launch checks below report only this call's launches
  if (!c->have_design || c->nk == 0) return PC_ESTATE;
  if (k < 0 || k >= c->nk || ncols > c->nk * c->m) return PC_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  if (c->prm.precision == PC_MIXED) {
    // the mixed form's operator: FP32 vectors, split-BF16 tensor-core products, SI on return
    const long long n = (long long)ncols * 3 * c->N;
    float2* xf = (float2*)c->blk[3];
    float2* af = (float2*)c->blk[4];
    float2* of = (float2*)c->blk[5];
    int rc = launch_d2f((const double2*)x, xf, n, 1.0, s);
    if (!rc) rc = apply_fp32(c, xf, af, of, ncols, ncols, k, s);
    if (!rc) rc = launch_convert_f2d(af, (double2*)ax, n, s);
    if (!rc) rc = launch_convert_f2d(of, (double2*)ox, n, s);
    if (!rc) rc = launch_scale_d2((double2*)ax, n, c->sA, s);
    if (!rc) rc = launch_scale_d2((double2*)ox, n, c->sO, s);
    return rc;
  }
  const double two_pi = 2.0 * M_PI;
  const double epi = two_pi * two_pi * c->V * c->V;  // SI: (2 pi V)^2
  return apply_fp64(c, (const double2*)x, (double2*)ax, (double2*)ox, ncols, ncols, c->Q + 3LL * k, epi, 1.0,
                    c->Ed, c->Sd, s);
}

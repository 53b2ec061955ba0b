// Internal launch interfaces shared by the translation units of the library.
#pragma once
#include "common.cuh"

// A phase accepted by pc_create: rho > 0, E > 0 (both finite), -1 < nu < 0.5.
bool pc_material_ok(const pc_material& m);
// Concurrent k groups of a context's mixed form, set before pc_set_kpoints (phononic.cu).
int pc_internal_set_groups(pc_ctx* c, int groups);

struct MaterialConsts {
  int law;             // PC_LAW_COMPLIANCE | PC_LAW_YOUNG
  double E0, E1, nu0, nu1;  // Young's modulus and Poisson ratio of phase0 / phase1 (PC_LAW_YOUNG)
  double penal;
  double rho0, rho1;   // mass density of phase0 / phase1
  double f1_0, f1_1;   // bulk compliance (1-2nu)/E
  double f2_0, f2_1;   // shear compliance (1+nu)/E
};

struct SetupArgs {
  const double* rho;
  int n0, n1, n2, M;
  double V;
  MaterialConsts mc;
  double* fields;   // 3 x ne
  double* dchi;     // ne
  double* chi;      // ne
  double* dfc;      // 2 x ne: d f1 / d chi, d f2 / d chi per element
  double* chi_mean; // 1
  double2* t1;      // 3 x n0 x n1 x L
  double2* t2;      // 3 x n0 x L x L
  double2* sfac;    // 3 x L^3
  double2* T;       // 3 x N x N   (density, f1, f2), SI
  double2* W;       // 2 x N x N   inverses of the f1, f2 blocks, SI
  double2* gj;      // setup_gj_scratch(N): panels of the blocked Gauss-Jordan steps
  int* status;
};
long long setup_gj_scratch(int N);
int launch_setup(const SetupArgs& a, cudaStream_t s);

int device_sms();  // multiprocessors of the device (152 where it cannot be asked)

// Geometry needed on the device to form K_q = T (Q_k + g_q).
struct Geom {
  double T[9];  // reciprocal basis, row-major: K_i = sum_j T[i*3+j] * (Q_j + g_j)
  int M;
  int N;
};

// A selection of the vectors of a block: entry v of nvec stands for vector list[v] (per = 1) or
// list[v / per] * per + v % per (whole k-points, per = m), or for v itself without a list.
struct VecSel {
  const int* list = nullptr;
  int per = 1;
  __device__ __forceinline__ int operator()(int v) const {
    return !list ? v : (per == 1 ? list[v] : list[v / per] * per + v % per);
  }
};

// Complex GEMMs C[col][p] = alpha * sum_q A[p][q] B[col][q] (both operands K-contiguous) of the same
// shape but for their columns, nseg <= 3 in one launch.
template <typename R> struct GemmSeg {
  const typename cplx_t<R>::type* A;
  const typename cplx_t<R>::type* B;
  typename cplx_t<R>::type* C;
  int ncols;
  R alpha;
  VecSel sel = {};  // selected vectors of three columns each: column j of B and C is that of vector sel(j / 3)
  __device__ __forceinline__ long long column(long long j) const {
    return sel.list ? 3LL * sel((int)(j / 3)) + j % 3 : j;
  }
};
template <typename R>
int launch_gemms(int Mrows, int K, int lda, long long ldb, long long ldc, const GemmSeg<R>* seg, int nseg, cudaStream_t s);

// Operator pieces.  Vector blocks are [vec][3][N] complex, vec = k*m + j.
template <typename R>
int launch_strain(const typename cplx_t<R>::type* X, int nvec, int m, Geom g, const double* Q,
                  typename cplx_t<R>::type* E, cudaStream_t s, const float4* Kf = nullptr, VecSel sel = {});
// Stresses of nvec selected vectors (compact in Sig) into their columns of AX.
template <typename R>
int launch_epilogue(const typename cplx_t<R>::type* Sig, int nvec, int m, Geom g, const double* Q,
                    R c0, R c1, typename cplx_t<R>::type* AX, cudaStream_t s, const float4* Kf = nullptr, VecSel sel = {});
// Kf[k N + q] = FP32 wavevector (K_0, K_1, K_2, 0) of plane wave q at the k-th point of Q (nk points);
// the FP32 kernels above and below read it when given (it is ignored for FP64 data).
int launch_kvec_table(Geom g, const double* Q, int nk, float4* Kf, cudaStream_t s);

struct PrecRef {  // reference medium from the mean of chi (device scalar)
  double lam0, lam1, mu0, mu1, rho0, rho1;
  double f1_0, f1_1, f2_0, f2_1;  // compliance moduli (1-2nu)/E, (1+nu)/E of the phases
  double two_pi_sq_V_over_sA;
  double half_lref_V_over_sA;
  int ref_mode;       // 0: Lame constants linear in chi; 1: compliance linear in chi (the material law); 2: between
  double shift_scale; // weight of the mass term rho sigma
};
// k-points still iterated, kept on the device and counted on the host: klist the open k-points in
// order, vlist their unconverged vectors (k m + j), fresh the k-points that the last test locked, count
// {open, unconverged vectors, fresh, open ones above the tolerance}: an open k-point may have met it.
struct OpenSet {
  int *klist, *vlist, *fresh, *count;
  int* vpos;  // position of an open k-point's vector in vlist, or -1
};
// klist = all; ref (3 doubles) = 3 kappa and 2 mu of the preconditioner's reference medium and the factor of
// its shift, nondimensional.
int launch_open_all(OpenSet o, int nk, PrecRef pr, const double* chi_mean, double* ref, cudaStream_t s);
// Residuals of the nopen k-points of o.klist, then the convergence test: kdone, and the new lists.
template <typename R>
int launch_resnorm(const typename cplx_t<R>::type* AX, const typename cplx_t<R>::type* OX,
                   const R* lam, int nk, int m, int nb, int n3, double tol, double* rnorm,
                   int* active, int* kdone, OpenSet o, int nopen, cudaStream_t s, double* best = nullptr,
                   int* since = nullptr);
// The preconditioner W = P(R) on the ncol vectors of vlist, in two halves around the products S = T E of the
// compliance operators (T_f1 on stack 0, T_f2 on the others) with the strain stacks E; W, A W and Omega W = 0
// on the other vectors of the open k-points.
template <typename R>
int launch_prec_in(const typename cplx_t<R>::type* AX, const typename cplx_t<R>::type* OX, const R* lam, const int* vlist,
                   int ncol, int m, int nb, Geom g, const double* Q, const double* ref, typename cplx_t<R>::type* W,
                   typename cplx_t<R>::type* E, cudaStream_t s, const float4* Kf = nullptr);
template <typename R>
int launch_prec_out(const typename cplx_t<R>::type* S, const R* lam, const int* klist, const int* vpos, int nopen, int ncol,
                    int m, int nb, Geom g, const double* Q, const double* ref, typename cplx_t<R>::type* W,
                    typename cplx_t<R>::type* AW, typename cplx_t<R>::type* OW, cudaStream_t s, const float4* Kf = nullptr);
// dst[k] = src[k] in FP64 for the nsel k-points of list, `per` values each.
template <typename R>
int launch_store(const typename cplx_t<R>::type* src, double2* dst, const int* list, int nsel, long long per, cudaStream_t s);
template <typename R>
int launch_init_guess(typename cplx_t<R>::type* X, int nk, int m, Geom g, const double* Q, unsigned long long seed,
                      cudaStream_t s);

// Block operations of the eigensolver, batched over k.  A "block" is m vectors of n3 rows
// per k, base pointer + k * m * n3.
template <typename R> struct BlockList {
  const typename cplx_t<R>::type* p[3];
};
// A batch of small matrices of nel entries as its consumers read it: entry e of problem i is
// scale * sum_{t < nsplit} p[(i nsplit + t) nel + e], so that the row-split partial sums of a Gram
// product need no reduction launch of their own.
template <typename R> struct MatRef {
  typedef typename cplx_t<R>::type C2;
  const C2* p = nullptr;
  long long nel = 0;
  int nsplit = 1;
  R scale = 1;
  __device__ __forceinline__ C2 at(long long i, int e) const {
    const C2* q = p + i * nsplit * nel + e;
    C2 s = q[0];
    for (int t = 1; t < nsplit; ++t) s = cadd(s, q[t * nel]);
    return cscale(s, scale);
  }
  MatRef from(long long i) const {  // the problems from i on
    MatRef r = *this;
    r.p = p + i * nsplit * nel;
    return r;
  }
};
// Gram products of nk k-points (of klist, or all); problem i of the result is the i-th of them.  part:
// workspace of at most max_split partial results per problem; G: the reduced result, where the kernel
// reduces (FP64 and the CUDA-core FP32 kernel).
template <typename R>
int launch_gram(BlockList<R> A, int na, BlockList<R> B, int nb_, int nk, int m, int n3, R scale,
                typename cplx_t<R>::type* part, typename cplx_t<R>::type* G, MatRef<R>* out, cudaStream_t s,
                int* status = nullptr, const int* klist = nullptr, int max_split = 8);
template <typename R> struct UpdateArgs {
  const typename cplx_t<R>::type* in[3][3];  // [triplet][block]
  typename cplx_t<R>::type* out[3];
  int ntrip, nblk;
  int identity_last;   // out = in[last] + sum_{b<last} in[b] C_b
  MatRef<R> C;         // per problem: rows (nblk or nblk-1)*m, cols mout
  int cld;             // leading dimension (columns) of C
  const int* klist = nullptr;  // k-point of problem i (or i itself)
  int m, mout, n3, nk;
  long long in_kstride, out_kstride;  // elements per k (normally m*n3 / mout*n3)
  // optional second coefficient set over the same inputs: out2[t] = sum_b in[t][b] C2nd_b
  MatRef<R> C2nd;  // p = nullptr: none
  typename cplx_t<R>::type* out2[3] = {nullptr, nullptr, nullptr};
  int* status = nullptr;  // device status word (tensor-core kernels record a timeout there)
};
template <typename R> int launch_update(const UpdateArgs<R>& a, cudaStream_t s);
// Tensor-core versions for FP32 data (tall_tc.cu); g_tc_tall = 0 selects the CUDA-core kernels.
// Process-wide switches read by every launch, from any k-group thread.
extern std::atomic<int> g_tc_tall;
int launch_gram_tc(const float2* const A[3], int na, const float2* const B[3], int nbk, int nk, int m, int n3,
                   float scale, float2* part, int max_split, MatRef<float>* out, int* status, const int* klist,
                   cudaStream_t s);
int launch_update_tc(const UpdateArgs<float>& u, int* status, cudaStream_t s);

// Projected problems, one CTA per k: the pencil (GA, GO) of n <= 72 basis columns, unit-diagonal
// scaling, Cholesky of GO that drops dependent columns (pivots at or below drop_tol), reduction to
// standard form, cyclic Jacobi; the lowest m eigenvalues (at the k-point of klist, or the problem's own
// index) and their coefficients (n x m).  When cp is given, the conjugate-direction coefficients of the next
// iteration come from the same CTA (directions at or below pdir_abs dropped); when flops is given, the
// algorithmic flops of every problem solved are added to it (device counter).  scratch: global scratch of
// `stride` bytes, at least small_rr32_scratch(n) / small_rr64_scratch(n) and a multiple of 16, for each of `slots` problems;
// more problems than that take several launches.
// others: problems that other calls are solving meanwhile (launch_rules.h).
int launch_small_rr32(const MatRef<float>& GA, const MatRef<float>& GO, int n, int m, int nk, float drop_tol, const int* klist,
                      float* lam_out, float2* coef, float2* cp, float pdir_abs, int* status, double* flops,
                      void* scratch, long long stride, int slots, cudaStream_t s);
int launch_small_rr64(const MatRef<double>& GA, const MatRef<double>& GO, int n, int m, int nk, double drop_tol, const int* klist,
                      double* lam_out, double2* coef, double2* cp, double pdir_abs, int* status, void* scratch,
                      long long stride, int slots, long long others, cudaStream_t s);
long long small_rr32_scratch(int n);
long long small_rr64_scratch(int n);
// Cholesky-QR transform of the Gram matrices G (m x m).
template <typename R>
int launch_small_chol(const MatRef<R>& G, int m, int nk, R drop_tol, typename cplx_t<R>::type* T, cudaStream_t s);

int launch_convert_f2d(const float2* src, double2* dst, long long n, cudaStream_t s);

// Gap objective and adjoint.
struct GapArgs {
  const double* lam;     // nk x nb, nondimensional
  int nk, nb, n_lower, mode;
  double lref;           // lambda_phys = lam * lref
  double rel_tol;
  double ks_beta;        // smooth (KS) gap: sharpness on omega / omega_ref (mode PC_GAP_KS_INTERNAL)
  const double* w_user;  // for PC_GRAD_ALLBANDS
  double* gap_out;
  double* weights;       // nk x nb, dG / dlambda_phys
  int* pairs;            // list of (k*nb + b) with non-zero weight
  int* npairs;
};
int launch_gap(const GapArgs& a, cudaStream_t s);
#define PC_GAP_KS_INTERNAL 3  // mode of GapArgs for pc_gap_ks_and_grad

struct AdjointArgs {
  const double2* theta;  // [vec][3][N], nondimensional eigenvectors (X' with X'^H Omega' X' = I)
  const double2* sig;    // [6][nvec][N], W_s E_s of theta (SI W, strain without 2 pi)
  const double* lam;     // nk x nb nondimensional
  const double* weights; // nk x nb physical
  const int* pairs;
  const int* npairs;
  int max_pairs;
  int nk, nb, m, N, M, n0, n1, n2;
  double lref;           // physical lambda scale
  double inv_sO;         // |theta_phys|^2 = |X'|^2 / sO
  double d_rho;
  const double* dfc;     // 2 x ne: d f1 / d chi and d f2 / d chi per element
  double two_pi_V_sq;    // (2 pi V)^2 over the square of the stresses' scale
  double w_scale, w_inv; // power of two that the weights are multiplied by, and its inverse
  double ve;             // element volume
  const double* dchi;
  void* t2;              // scratch: max_pairs x 9 x M2 x n1 x n2 complex (FP64 or FP32)
  const void* phases;    // launch_adj_phases
  void* part;            // scratch: room for kAdjChunksMax x 3 x ne FP64 sums, or twice as many in FP32
  double* grad;
};
constexpr int kAdjChunksMax = 32;  // pair chunks of the adjoint's reduction
// Phases of the synthesis for a grid and cutoff: M (n0 + n1 + n2) complex values in the adjoint's precision.
int launch_adj_phases(int M, const int n[3], bool fp32, void* ph, cudaStream_t s);
// fp32: synthesis in FP32 (mixed form); the weighted sum is accumulated in FP64 either way.
int launch_adjoint(const AdjointArgs& a, bool fp32, cudaStream_t s);
// Dynamic shared memory allowed for the adjoint's field-synthesis kernel: the N coefficients of one
// eigenvector component, (2M+1)^2 n2 sums along axis 2 and (2M+1)(n1 + n2) phases, of which it stages
// M (n1 + n2); complex values of the form's precision.  Grids and cutoffs above kAdjointStagingMax are refused.
size_t adjoint_staging_bytes(int M, int n1, int n2, bool fp32);
constexpr size_t kAdjointStagingMax = 200 * 1024;

// omega[k][b] = sqrt(max(lam_m[k][b] * lref, 0)) and lam_nd[k][b] = lam_m[k][b] for b < nb.
int launch_omega(const double* lam_m, int nk, int nb, int m, double lref, double* omega, double* lam_nd,
                 cudaStream_t s);
int launch_d2f(const double2* src, float2* dst, long long n, double scale, cudaStream_t s);
int launch_scale_d2(double2* x, long long n, double s, cudaStream_t st);

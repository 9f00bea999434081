// Shared definitions of the GB300 Richards solver: context, sparse/level structs,
// launch helpers, deterministic block reductions and the constitutive law.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "../../include/richards.h"
#include "fixpow.cuh"

namespace rich {

constexpr int kBlock = 256;          // threads per block of every elementwise kernel
constexpr int kNumSM = 152;          // GB300 SM count (2 dies x 76)
constexpr int kRedBlocks = 8 * kNumSM;  // fixed grid of the reduction kernels (deterministic order)

void set_cuda_error(cudaError_t e, const char* where);

#define RICH_CUDA(call)                                              \
  do {                                                               \
    cudaError_t e_ = (call);                                         \
    if (e_ != cudaSuccess) {                                         \
      ::rich::set_cuda_error(e_, #call);                             \
      return RICH_ECUDA;                                             \
    }                                                                \
  } while (0)

#define RICH_CHECK(...)                  \
  do {                                   \
    int s_ = (__VA_ARGS__);              \
    if (s_ != RICH_OK) return s_;        \
  } while (0)

// Every kernel launch is followed by RICH_LAUNCH_CHECK, which also counts it.
void count_launch();
void count_launches(long long k);  // k may be negative (launches recorded into a graph)
#define RICH_LAUNCH_CHECK()        \
  do {                             \
    ::rich::count_launch();        \
    RICH_CUDA(cudaGetLastError()); \
  } while (0)

// Optional live timing of one named kernel: when its name matches the profiling
// target, CUDA events are recorded around its launches on the launching stream.
// Moves the start of the open timed launch to now (work done on the stream since
// it opened, e.g. a one-time layout, is not charged to the launch).
void prof_restart(cudaStream_t st);
struct ProfScope {
  bool on;
  cudaStream_t st;
  double bytes, flops;
  ProfScope(const char* name, cudaStream_t s, double algorithmic_bytes, double algorithmic_flops = 0.0);
  ~ProfScope();
};

inline int grid_for(long long n, int block = kBlock) {
  long long g = (n + block - 1) / block;
  if (g < 1) g = 1;
  if (g > 2147483647LL) g = 2147483647LL;
  return (int)g;
}
inline int red_grid(long long n) {
  long long g = (n + kBlock - 1) / kBlock;
  if (g > kRedBlocks) g = kRedBlocks;
  if (g < 1) g = 1;
  return (int)g;
}

struct SoilP {
  double alpha, beta, ts, tr, a, gamma, ks, rho_phi;
  double cs, cds, cdk, cka;   // alpha (ts - tr), alpha beta (ts - tr), a gamma, ks a
  unsigned long long qb, qg;  // beta, gamma for fixpow_exp2; both 0: pow() throughout
};

// The fixed-point powers serve exponents in (0, 32) and constants whose sums with the
// powers (below 2^960) have a normal reciprocal; other soils take pow().
inline SoilP soil_params(const rich_soil* s) {
  SoilP p{s->alpha, s->beta, s->theta_s, s->theta_r, s->a, s->gamma, s->ks_const, s->rho_phi};
  p.cs = s->alpha * (s->theta_s - s->theta_r);
  p.cds = s->alpha * s->beta * (s->theta_s - s->theta_r);
  p.cdk = s->a * s->gamma;
  p.cka = s->ks_const * s->a;
  p.qb = fixpow_exponent(s->beta);
  p.qg = fixpow_exponent(s->gamma);
  auto normal = [](double v) { return v >= 1e-280 && v <= 1e280; };
  if (!p.qb || !p.qg || !normal(s->alpha) || !normal(s->a)) p.qb = p.qg = 0;
  return p;
}

struct GridP {
  int nx, ny, nz;
  int nzs;           // layers per stacked problem (nz unless a batch stacks several problems along z)
  long long n;
  double inv_h[3];   // 1/h_d
  double inv_h2[3];  // 1/h_d^2
  double half_h2[3]; // 1/(2 h_d^2)
  double twice_h2[3];  // 2/h_d^2
  double half_hz;    // 1/(2 h_z)
  void set_spacing(const double h[3]) {
    for (int d = 0; d < 3; ++d) {
      inv_h[d] = 1.0 / h[d];
      inv_h2[d] = 1.0 / (h[d] * h[d]);
      half_h2[d] = 0.5 * inv_h2[d];
      twice_h2[d] = 2.0 * inv_h2[d];
    }
    half_hz = 0.5 * inv_h[2];
  }
};

struct BCP {
  int kind[6];
  double value[6];
  const double* field[6];  // per-cell Dirichlet values (ghost pressures of an interface face), or nullptr
  const double* gks[6];    // interface faces: per-cell K_s of the ghost cells, or nullptr (soil ks)
};

// Cell spacing of a grid: the explicit h[d] where given, else l / (n + 1).
inline void grid_spacing(const rich_grid* g, double h[3]) {
  h[0] = g->h[0] > 0 ? g->h[0] : g->lx / (g->nx + 1);
  h[1] = g->h[1] > 0 ? g->h[1] : g->ly / (g->ny + 1);
  h[2] = g->h[2] > 0 ? g->h[2] : g->lz / (g->nz + 1);
}

// Index of the boundary cell (i, j, k) in the per-cell arrays of face f.
__device__ __forceinline__ long long face_index(int f, int i, int j, int k, int nx, int ny) {
  int axis = f >> 1;
  return axis == 2 ? (long long)i + (long long)nx * j
                   : (axis == 1 ? (long long)i + (long long)nx * k : (long long)j + (long long)ny * k);
}

// Dirichlet value of face f at the boundary cell (i, j, k).
__device__ __forceinline__ double bc_value(const BCP& bc, int f, int i, int j, int k, int nx, int ny) {
  const double* fv = bc.field[f];
  if (!fv) return bc.value[f];
  return fv[face_index(f, i, j, k, nx, ny)];
}

template <class T>
struct Csr {
  int nrows = 0, ncols = 0;
  long long nnz = 0;
  int* rowptr = nullptr;
  int* col = nullptr;
  T* val = nullptr;
};

// SELL-C-sigma copy of a CSR matrix for the coarse-level row operations: rows are
// sorted by decreasing length within windows of kSellSigma rows and cut into slices
// of kSellC = 32 (one warp, one thread per row); slice s is stored column by column,
// slot sptr[s] + 32 j + t holding the j-th entry of row perm[32 s + t] (value and
// column), or a zero with column 0 past the end of that row.  Loads of a slice are
// coalesced and a row needs no cross-lane reduction.
constexpr int kSellC = 32;
constexpr int kSellSigma = 1024;
constexpr int kSellMinRows = 2048;
struct Sell {
  int nrows = 0, nslice = 0;
  long long slots = 0;
  int* sptr = nullptr;      // nslice + 1 slot offsets
  int* perm = nullptr;      // 32 nslice rows, -1 past nrows
  int* col = nullptr;       // slots
  double* val = nullptr;    // values for an FP64 hierarchy
  float* val32 = nullptr;   // values for an FP32 hierarchy (MIXED)
  bool built() const { return sptr != nullptr; }
};

// Galerkin refresh by product lists: entry q of C = A B is the sum of a[x] * b[y] over
// its pairs (x, y), in A-entry order.  Entries are ranked by their number of pairs within
// windows of kSellSigma and cut into slices of 32, the pairs of a slice stored column by
// column as in Sell (slot sptr[s] + 32 j + t: pair j of entry perm[32 s + t], x = -1 past its
// end), so that a warp reads its pairs coalesced and its threads end together.
struct ProdList {
  long long np = 0;            // pairs (= scalar products of C = A B)
  int nslice = 0;
  int* perm = nullptr;         // 32 nslice entries of C, -1 past the last
  long long* sptr = nullptr;   // nslice + 1 slot offsets
  int2* pairs = nullptr;
  bool built() const { return pairs != nullptr; }
};

// One level of the AMG hierarchy.  Level 0 holds the diffusion matrix of the
// finest grid; levels 1.. hold Galerkin products.  FP32 copies exist in MIXED mode.
struct Level {
  int n = 0;
  Csr<double> A;
  float* A32 = nullptr;            // values of A in FP32 (pattern of A)
  double* dinv = nullptr;          // 1 / sum_j |a_ij|
  float* dinv32 = nullptr;
  int* agg = nullptr;              // aggregate of each node (levels with a coarser level)
  Csr<double> P, R, AP;            // to the next level; AP = A P (pattern kept for refresh)
  int* u_ap = nullptr;             // products per row of A P and of R (A P) (refresh kernels' split)
  int* u_rap = nullptr;
  float* P32 = nullptr;            // values of P/R in FP32
  float* R32 = nullptr;
  float* AP32 = nullptr;           // values of A P in FP32 (MIXED-precision refresh)
  ProdList pl_ap, pl_rap;          // product lists of A P and R (A P), built at the first refresh
  Sell sA, sP, sR;                 // SELL-C-sigma copies (levels with >= kSellMinRows rows)
  bool pl_tried = false;
  int mis_rounds = 0;
  double omega = 0.0;
  // V-cycle work vectors, typed by the hierarchy precision (double or float)
  void* x = nullptr;
  void* b = nullptr;
  void* r = nullptr;
  void* t = nullptr;
};

// Finest level of the V-cycle in stencil form: the diffusion matrix is symmetric
// with non-negative face weights w (coupling -w), so four arrays hold it:
// diagonal, and the +x, +y, +z face weights of each cell (0 on the boundary).
template <class T>
struct Stencil4 {
  T* diag = nullptr;
  T* wx = nullptr;
  T* wy = nullptr;
  T* wz = nullptr;
  T* dinv = nullptr;  // 1 / (diag + sum of the six face weights), the l1-Jacobi scaling
};

// Finest level of the l1-Jacobi V-cycle, scaled symmetrically: with s = l1^-1/2 per cell
// (l1 the row's l1 norm) and A' = s A s, x = s y and b' = s b, the sweep
// x <- x + l1^-1 (b - A x) is y <- b' + (I - A') y: one multiply-add per entry and no
// other FP64 operation, and the first sweep from zero is y = b' itself.  g is the diagonal
// of I - A' and gd that of -A', wx wy wz the face weights scaled from both sides, q = 1 / s.
template <class T>
struct ScaledSt {
  T* g = nullptr;
  T* gd = nullptr;
  T* wx = nullptr;
  T* wy = nullptr;
  T* wz = nullptr;
  T* s = nullptr;
  T* q = nullptr;
};

// Launch shape of the structured-grid kernels: one block row per (j, k) grid line,
// blockIdx.y tiles the x direction; no 64-bit division per thread.
constexpr int kLineThreads = 128;
inline dim3 line_grid(const GridP& g) {
  return dim3((unsigned)((long long)g.ny * g.nz), (unsigned)((g.nx + kLineThreads - 1) / kLineThreads), 1);
}

struct Hierarchy {
  Stencil4<double> st64;
  Stencil4<float> st32;
  ScaledSt<double> sc64;
  ScaledSt<float> sc32;
  bool scaled = false;            // the finest level runs on sc64 / sc32 (l1-Jacobi, more than one level)
  std::vector<Level> lv;
  int nlev = 0;
  int cn = 0;                     // coarsest size
  double* cdense = nullptr;       // coarsest matrix, dense, then its inverse (cn x cn)
  float* cinv32 = nullptr;
  double* cwork = nullptr;        // blocked Gauss-Jordan work: panel rows, old panel columns, panel inverse
  rich_amg_opts opts{};
  bool built = false;
  bool dense = true;              // coarsest level by dense inverse (else kCoarseSweeps l1-Jacobi sweeps)
  cudaGraphExec_t gj_exec = nullptr;  // the coarsest inverse (one launch per pivot) as one graph
  long long gj_nodes = 0;
  // the V-cycle as one graph (opts.graph): captured at its second application,
  // reading the level-0 right-hand side buffer and leaving its result at vc_out
  cudaGraphExec_t vc_exec = nullptr;
  long long vc_nodes = 0;
  void* vc_out = nullptr;
  int vc_calls = 0;
  bool vc_off = false;            // capture failed: direct launches for this hierarchy
  // FCG's iterations as one graph (a WHILE loop, solve.cu); kernels per iteration.  The number
  // of stacked problems is part of a captured loop: [0] one problem, [1] the batch's nbatch
  // (a batch context reaches both: its own step, and a lone solve or step over the stack).
  cudaGraphExec_t fcg_exec[2] = {nullptr, nullptr};
  long long fcg_nodes[2] = {0, 0};
  bool fcg_off = false;
  // one-level additive Schwarz (precond = RICH_PRECOND_AS): ILU(0) diagonals and
  // subdomain solutions (hierarchy precision), FP32 staging of r and z in MIXED
  void* asD = nullptr;
  void* asZ = nullptr;
  float* asR32 = nullptr;
  float* asZ32 = nullptr;
};

constexpr int kStallWindow = 30;        // FCG iterations per stagnation test (krylov.stall)
constexpr int kMaxCoarseDense = 8192;  // largest coarsest level inverted densely
constexpr int kCoarseSweeps = 8;       // l1-Jacobi sweeps on a stalled (larger) coarsest level

struct KrylovWork {
  long long n = 0;
  int m = 0;
  double* V = nullptr;  // (m+1) x n
  double* Z = nullptr;  // m x n
  double* x = nullptr;
  double* r = nullptr;
  double* p = nullptr;
  double* q = nullptr;
  double* z = nullptr;
  double* w = nullptr;
  double* hcoef = nullptr;  // device coefficients (m+1)
  double* gram = nullptr;   // V^T V of FGMRES' basis (64 x 64)
  unsigned* peak = nullptr; // high words of the basis vectors' largest entries (64)
  void* fcg = nullptr;      // FCG's scalars on the device (FcgDev)
  void* fcg_out = nullptr;  // and what the host reads of them (pinned)
  int fail_reason = 0;      // last failure: 0 none, FCG 1 maxit, 2 (p, J p) <= 0, 3 residual growth;
                            // 4 stagnation (an FCG window or an FGMRES restart cycle, krylov.stall)
};

}  // namespace rich

struct rich_ctx {
  rich::GridP g{};
  rich::SoilP soil{};
  rich::BCP bc{};
  int kmean = 0;
  int prec = 0;
  cudaStream_t st = nullptr;
  int device = 0;
  double* ks = nullptr;        // per-cell K_s or nullptr
  // K, K' and s' at the last p of a constitutive pass or a storing residual
  double* K = nullptr;
  double* dK = nullptr;
  double* dS = nullptr;
  // stencils (7n)
  double* J7 = nullptr;
  double* A7 = nullptr;
  bool have_jac = false;
  bool a0_fresh = false;       // finest CSR values match A7
  // finest-level CSR pattern (built at create)
  rich::Csr<double> A0;
  rich::Hierarchy H;
  rich::KrylovWork kw;
  // reductions: partial sums per block and device scalars
  double* partials = nullptr;  // kRedBlocks * 64
  double* dsc = nullptr;       // device scalars (256)
  double* hsc = nullptr;       // pinned host mirror (128)
  unsigned* ticket = nullptr;  // finished blocks per segment of a reduction (32, zero between launches)
  int* iflag = nullptr;        // device int flags (16)
  int* hflag = nullptr;        // pinned host (16)
  // Newton work
  double* s_old = nullptr;
  double* F = nullptr;
  double* Ft = nullptr;
  double* d = nullptr;
  double* ptrial = nullptr;
  double* rhs = nullptr;
  double* pbuf = nullptr;      // device p for rich_step_host
  double* psave = nullptr;     // p at the start of a substep (time-step control)
  int nbatch = 1;              // problems stacked along z (rich_create_batch)
  double* bc_fields[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};  // owned per-cell BC values
  double* bc_gks[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};     // owned ghost K_s (interfaces)
  bool amg_ever = false;
};

namespace rich {

// ---------------------------------------------------------------- device helpers

// Constitutive law, eqs. (s(p)), (K(p)) and (derivativeofcoefficients) of Sec. 2-3, for
// p < 0 outside the fixed-point domain (|p| beyond 2^+-30, unusual soils); |p|^(x-1) =
// |p|^x / |p|.
struct Law {
  double S, dS, K, dK;
};
static __device__ __noinline__ Law law_general(double ap, double ks, double alpha, double beta, double ts, double tr,
                                               double a, double gamma) {
  const double pb = pow(ap, beta);
  const double pg = pow(ap, gamma);
  const double r_ap = 1.0 / ap;
  const double r_s = 1.0 / (alpha + pb);
  const double r_k = 1.0 / (a + pg);
  return Law{alpha * (ts - tr) * r_s + tr, alpha * beta * (pb * r_ap) * (ts - tr) * (r_s * r_s), ks * a * r_k,
             a * gamma * ks * (pg * r_ap) * (r_k * r_k)};
}
__device__ __forceinline__ Law law_general(double p, double ks, const SoilP& so) {
  return law_general(-p, ks, so.alpha, so.beta, so.ts, so.tr, so.a, so.gamma);
}

// Whether p is negative with |p| in the domain of the fixed-point powers (sign bit set,
// binary exponent in [-30, 29]; integer tests: no FP64 compare).
__device__ __forceinline__ bool law_fast(double p, const SoilP& so) {
  constexpr unsigned lo = 0x80000000u | ((unsigned)(1023 - kFixPowExp) << 20);
  return so.qb != 0 && (unsigned)__double2hiint(p) - lo < ((unsigned)(2 * kFixPowExp) << 20);
}
__device__ __forceinline__ long long law_log(double p) {
  return fixpow_log2((unsigned long long)__double_as_longlong(p) & 0x7fffffffffffffffull);
}

// K(p) (and, below, the rest of the law) from the fixed-point powers: the sums, one
// reciprocal each and the products are all that runs in FP64 (K alone 6 operations, the
// whole law 23 against about 95 through log()/exp() and divisions).  FP64 pipe bound
// both ways: the law of 2.1M cells took 370 us before and takes 94.
__device__ __forceinline__ double conductivity_only(double p, double ks, double ksa, const SoilP& so) {
  if (law_fast(p, so)) return ksa * fast_rcp(so.a + fixpow_exp2(law_log(p), so.qg));
  return p < 0.0 ? law_general(p, ks, so).K : ks;
}
__device__ __forceinline__ double conductivity_only(double p, double ks, const SoilP& so) {
  return conductivity_only(p, ks, ks * so.a, so);
}
__device__ __forceinline__ double saturation_only(double p, const SoilP& so) {
  if (law_fast(p, so)) return fma(so.cs, fast_rcp(so.alpha + fixpow_exp2(law_log(p), so.qb)), so.tr);
  return p < 0.0 ? law_general(p, 1.0, so).S : so.ts;
}

__device__ __forceinline__ void constit(double p, double ks, const SoilP& so, double& S, double& dS,
                                        double& K, double& dK) {
  if (law_fast(p, so)) {
    const long long y = law_log(p);
    const double pb = fixpow_exp2(y, so.qb), pg = fixpow_exp2(y, so.qg);
    const double r_ap = fast_rcp(-p), r_s = fast_rcp(so.alpha + pb), r_k = fast_rcp(so.a + pg);
    S = fma(so.cs, r_s, so.tr);
    dS = (so.cds * (pb * r_ap)) * (r_s * r_s);
    K = (ks * so.a) * r_k;
    dK = (so.cdk * ks) * (pg * r_ap) * (r_k * r_k);
  } else if (p < 0.0) {
    const Law w = law_general(p, ks, so);
    S = w.S;
    dS = w.dS;
    K = w.K;
    dK = w.dK;
  } else {
    S = so.ts;
    dS = 0.0;
    K = ks;
    dK = 0.0;
  }
}

// The mean used on the faces normal to axis: a split code (RICH_KMEAN_SPLIT) takes
// its horizontal mean on the x and y faces and its vertical mean on the z faces.
__host__ __device__ __forceinline__ int axis_mean(int kmean, int axis) {
  if (kmean & RICH_KMEAN_SPLIT_FLAG) return axis == 2 ? (kmean & 0xF) : ((kmean >> 4) & 0xF);
  return kmean;
}
inline bool kmean_valid(int kmean) {
  if (kmean >= 0 && kmean <= 3) return true;
  if ((kmean & ~0x1FF) != 0 || !(kmean & RICH_KMEAN_SPLIT_FLAG)) return false;
  return ((kmean >> 4) & 0xF) <= 3 && (kmean & 0xF) <= 3;
}

// Whether the upstream mean takes the upper cell, p_U - p_L >= 0, for dp = p_L - p_U
// (an integer test: sign bit or zero).
__device__ __forceinline__ bool dp_upstream(double dp) {
  const int hi = __double2hiint(dp);
  return hi < 0 || (hi | __double2loint(dp)) == 0;
}

// 1/q: three FP64 operations where q's exponent leaves room, else a division.
__device__ __forceinline__ double safe_rcp(double q) {
  const unsigned e = ((unsigned)__double2hiint(q) >> 20) & 0x7ffu;
  return e - 123u < 1800u ? fast_rcp(q) : 1.0 / q;
}

// Warp/block sum of NQ doubles in a fixed order; result valid in thread 0.
template <int NQ>
__device__ __forceinline__ void block_sum(double (&v)[NQ]) {
  __shared__ double sh[NQ][kBlock / 32];
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
  }
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) sh[q][wid] = v[q];
  }
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      double t = lane < kBlock / 32 ? sh[q][lane] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
      v[q] = t;
    }
  }
}

__device__ __forceinline__ double block_max(double v) {
  __shared__ double shm[kBlock / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) shm[wid] = v;
  __syncthreads();
  if (wid == 0) {
    double t = lane < kBlock / 32 ? shm[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t = fmax(t, __shfl_down_sync(0xffffffffu, t, o));
    v = t;
  }
  return v;
}

// ---------------------------------------------------------------- host helpers (blas.cu)

// Sum nq quantities of per-block partials (partials[q*nb + b]) into dst[q] (device), fixed order.
int finish_sums(rich_ctx* c, const double* partials, int nb, int nq, double* dst);
int finish_max(rich_ctx* c, const double* partials, int nb, double* dst);
int fetch_scalars(rich_ctx* c, const double* dsrc, int count, double* host);
int scan_exclusive_int(rich_ctx* c, const int* in, int* out, long long n);         // out[n] = total
int scan_exclusive_ll(rich_ctx* c, const long long* in, long long* out, long long n);
int scan_exclusive_int_ll(rich_ctx* c, const int* in, long long* out, long long n);
int dot(rich_ctx* c, const double* x, const double* y, long long n, double* dst_dev);
int nrm2sq(rich_ctx* c, const double* x, long long n, double* dst_dev);

// Device memory is stream-ordered: cudaMallocAsync / cudaFreeAsync on the
// stream of the context being worked on, so allocating or freeing never waits
// for the work of other streams (the request server runs several contexts at
// once).  Every entry point that may allocate names its stream with an
// AllocStream guard; outside one the legacy default stream is used, which is
// ordered with every blocking stream.  Freed blocks stay in the device's pool
// for reuse (release threshold raised once per device, see pool_setup).
extern thread_local cudaStream_t t_alloc_stream;
struct AllocStream {
  cudaStream_t prev;
  explicit AllocStream(cudaStream_t s) : prev(t_alloc_stream) { t_alloc_stream = s; }
  ~AllocStream() { t_alloc_stream = prev; }
};
void pool_setup();         // keeps freed device memory in the current device's pool
void pool_trim();          // returns the pool's unused memory (before free-memory queries)
size_t pool_slack();       // bytes the pool holds beyond what is in use
void* pinned_get();        // a 2 KB pinned host block from a process-wide free list
void pinned_put(void* b);  // back to the list (never cudaFreeHost: that synchronises the device)
constexpr size_t kPinnedBlock = 2048;

template <class T>
int dalloc(T** p, long long count) {
  if (count <= 0) count = 1;
  pool_setup();
  cudaError_t e = cudaMallocAsync((void**)p, sizeof(T) * (size_t)count, t_alloc_stream);
  if (e != cudaSuccess) {
    set_cuda_error(e, "cudaMallocAsync");
    *p = nullptr;
    return RICH_ENOMEM;
  }
  return RICH_OK;
}
template <class T>
void dfree(T*& p) {
  if (p) cudaFreeAsync((void*)p, t_alloc_stream);
  p = nullptr;
}

// physics.cu
int constit_eval(rich_ctx* c, const double* p);
// Phi(p) into F.  Newton's form also stores K, K' and s' for the Jacobian at this p and sums
// the round-off scale.  s_init, if not NULL: s_old is not read, s(p) stands in for it (Phi at
// the start of a step) and is written there.
// norms: the sums, per problem when nseg > 1 (the grid stacks nseg problems along z), are
// left at dsc[q * nseg + s] and in the pinned mirror hsc (quantity q: 0 ||F||^2, 1 ||F||_inf,
// 2 ||term magnitudes||^2, Newton's form only), valid once the stream has been waited for.
int residual_eval(rich_ctx* c, const double* p, const double* s_old, double dt, double* F, bool want_norms,
                  bool newton = false, double* s_init = nullptr, int nseg = 1);
// Waits for the context's stream and returns the first `count` scalars of the pinned mirror.
int wait_scalars(rich_ctx* c, int count, double* host);
// constit_current: the context's K, K', s' already hold the values of this p (the last
// storing residual was at the same pressure).
// J7b, A7b, if not NULL, receive copies of the two stencils.
int jacobian_eval(rich_ctx* c, const double* p, double dt, bool constit_current = false, double* J7b = nullptr,
                  double* A7b = nullptr);
int stencil_apply(rich_ctx* c, const double* A7, const double* x, double* y);
int refresh_a0_values(rich_ctx* c);

// amg_setup.cu
int amg_build(rich_ctx* c, const rich_amg_opts* o);
int amg_refresh(rich_ctx* c);
int amg_update_fine(rich_ctx* c);
void amg_free(rich_ctx* c);

// One problem's outcome of an FCG solve (reason: 0 converged, else KrylovWork::fail_reason).
struct FcgResult {
  double rn, bn;
  int it, reason;
};
int fcg_run(rich_ctx* c, int S, const double* b, double* x, const rich_krylov_opts* o, FcgResult* res);

// Keeps the stream busy for a number of GPU clocks (the loop ends by itself).
void gpu_delay(cudaStream_t st, long long cycles);

// blas.cu: whether a profiling target is set (the autotuner then stays off)
bool profiling_active();

// schwarz.cu
int as_setup(rich_ctx* c);   // allocate (first call) and factor every subdomain of the current A_aux
int as_apply(rich_ctx* c, const double* r, double* z);
void as_free(rich_ctx* c);

// sell.cu: SELL-C-sigma copies of the coarse-level matrices
int sell_build(rich_ctx* c, const Csr<double>& M, Sell& S);  // pattern; nothing below kSellMinRows rows
int sell_fill(rich_ctx* c, const Csr<double>& M, const double* val, Sell& S);  // values, M's entry order
int sell_fill(rich_ctx* c, const Csr<double>& M, const float* val, Sell& S);
void sell_free(Sell& S);

// solve.cu
int autotune_table(char* buf, int cap);
int autotune_load(const char* text);
int vcycle_apply(rich_ctx* c, const double* r, double* z);
int krylov_run(rich_ctx* c, const double* b, double* x, const rich_krylov_opts* o, rich_krylov_stats* st);

}  // namespace rich

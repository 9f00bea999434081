// Residual evaluation that allocates nothing (rich_residual_noalloc).
//
// Some callers cannot call cudaMalloc at the point where they need a residual:
// a serving loop that runs with a fixed, pre-reserved device memory budget, code
// that must not trigger the implicit device synchronisation a fresh allocation
// can cause, or an embedding application whose allocator owns all device memory.
// For them this entry point needs no context and no allocation: the caller
// passes the inputs and the output buffer, the block partial sums of the norms
// live in a fixed file-scope device array, and the constitutive values of each
// cell's neighbours are recomputed or shared on chip instead of being stored
// (the kernels of residual.cuh; 97 x 65 x 49 cells, harmonic mean: 348 us when
// every cell evaluated seven laws through log()/exp(), 114 now).
//
// The scratch array holds 2 partial sums for each of at most kNoAllocMaxBlocks
// blocks.  Grids up to kNoAllocMaxCells = 134,217,728 cells (512^3) are accepted;
// larger ones return RICH_ELIMIT.  The array (39 kB) stays resident on every
// device that loads the library until the process exits.  All calls share it:
// every call rewrites all the partials it reads, so nothing carries over between
// calls, but calls that overlap on the GPU (different streams, or different host
// threads) race on it and must be serialised by the caller.
#include <mutex>

#include "residual.cuh"

namespace rich {

constexpr long long kNoAllocMaxCells = 134217728;
constexpr int kNoAllocMaxBlocks = 16 * kNumSM;
constexpr int kNoAllocSlots = 2 * kNoAllocMaxBlocks + 8;  // partials, then the two results

static __device__ __align__(256) double g_noalloc_scratch[kNoAllocSlots];

// One block: sum / max of the nb partials in block order; results at slots 2*max, 2*max+1.
__global__ void k_residual_noalloc_finish(int nb, double* __restrict__ scratch) {
  double v[1] = {0.0};
  double m = 0.0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    v[0] += scratch[b];
    double a = scratch[kNoAllocMaxBlocks + b];
    m = (a > m || a != a) ? a : m;
  }
  block_sum<1>(v);
  m = block_max(m);
  if (threadIdx.x == 0) {
    scratch[2 * kNoAllocMaxBlocks] = v[0];
    scratch[2 * kNoAllocMaxBlocks + 1] = m;
  }
}

// Device address of the scratch array, looked up once per device with that
// device current (in host code the symbol itself is only a host-side stand-in).
static std::mutex g_noalloc_mu;
static double* g_noalloc_ptr[64] = {nullptr};

static int noalloc_scratch(double** out) {
  int dev = 0;
  RICH_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return RICH_ELIMIT;
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    if (e != cudaSuccess) {
      set_cuda_error(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
      return RICH_ECUDA;
    }
    g_noalloc_ptr[dev] = (double*)ptr;
  }
  *out = g_noalloc_ptr[dev];
  return RICH_OK;
}

}  // namespace rich

using namespace rich;

extern "C" int rich_residual_noalloc(const rich_grid* grid, const rich_soil* soil, int kmean, const rich_bc* bc,
                                     const double* p_dev, const double* s_old_dev, double dt, double* F_dev,
                                     double* norms_host, void* stream) {
  if (!grid || !soil || !bc || !p_dev || !s_old_dev || !F_dev || !(dt > 0)) return RICH_EINVAL;
  if (grid->nx < 1 || grid->ny < 1 || grid->nz < 1 || !(grid->lx > 0 && grid->ly > 0 && grid->lz > 0) ||
      !(grid->h[0] >= 0.0 && grid->h[1] >= 0.0 && grid->h[2] >= 0.0))
    return RICH_EINVAL;
  if (!kmean_valid(kmean)) return RICH_EINVAL;
  for (int f = 0; f < 6; ++f)
    if (bc->kind[f] != RICH_BC_NOFLUX && bc->kind[f] != RICH_BC_DIRICHLET) return RICH_EINVAL;
  long long n = (long long)grid->nx * grid->ny * grid->nz;
  if (n > kNoAllocMaxCells) return RICH_ELIMIT;
  double* scratch = nullptr;
  RICH_CHECK(noalloc_scratch(&scratch));
  GridP g;
  g.nx = grid->nx;
  g.ny = grid->ny;
  g.nz = grid->nz;
  g.nzs = grid->nz;
  g.n = n;
  double h[3];
  grid_spacing(grid, h);
  g.set_spacing(h);
  const SoilP so = soil_params(soil);
  BCP b;
  for (int f = 0; f < 6; ++f) {
    b.kind[f] = bc->kind[f];
    b.value[f] = bc->value[f];
    b.field[f] = bc->value_field_dev[f];
    b.gks[f] = nullptr;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const ResPlan pl = residual_plan(g, 1, kNoAllocMaxBlocks);
  ResOut out{};
  if (norms_host) out = ResOut{scratch, kNoAllocMaxBlocks, nullptr, nullptr, nullptr};
  residual_launch<false>(pl, 1, st, g, so, b, kmean, p_dev, s_old_dev, soil->ks_field_dev, so.rho_phi / dt, F_dev,
                         nullptr, nullptr, nullptr, nullptr, out);
  RICH_LAUNCH_CHECK();
  if (norms_host) {
    k_residual_noalloc_finish<<<1, kBlock, 0, st>>>(pl.nb, scratch);
    RICH_LAUNCH_CHECK();
    double r[2];
    RICH_CUDA(cudaMemcpyAsync(r, scratch + 2 * kNoAllocMaxBlocks, 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
    RICH_CUDA(cudaStreamSynchronize(st));
    norms_host[0] = sqrt(r[0]);
    norms_host[1] = r[1];
    if (!std::isfinite(norms_host[0]) || !std::isfinite(norms_host[1])) return RICH_ENONFINITE;
  }
  return RICH_OK;
}

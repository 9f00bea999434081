// The residual Phi(p) in one kernel: constitutive law, face fluxes and norms (Sec. 2.1,
// eq. (dynamic_of_the_problem); the face form is described in physics.cu).  Shared by the
// context's residual (physics.cu) and the allocation-free one (noalloc.cu).
//
// Bound: the FP64 pipe (two operations per SM and clock against 21 bytes of HBM per SM and
// clock; the 24 bytes a cell needs are 7 us of the 2.1M-cell grid, its FP64 work 80).  So
// the law's powers run on the integer pipe (fixpow.cuh), K is evaluated once per cell and
// shared through shared memory instead of a pass over memory, the two cells of a
// horizontal face compute its mean flux with four operations each, and a vertical face is
// computed once, by the thread that marches its column.  128^3, upstream mean, norms read
// back: 710 us as a law pass, a face pass and three single-block sums, 184 us here (38 FP64
// operations per cell against 64 to 95); 16^3: 55 to 23 us.
//
// A face's flux is the same number seen from either cell (t = k (p_L - p_U), exactly
// negated by the difference's antisymmetry), and every variant orders a cell's sum the
// same way, so Phi does not depend on the tiling or on where a grid is split.
#pragma once

#include "common.cuh"

namespace rich {

constexpr int kResThreads = 256;               // threads of a tile (tx * ty)
constexpr int kResHalo = 3 * (kResThreads + 2);  // (tx + 2) (ty + 2) at most (tx = 1 or 256)
constexpr int kCellThreads = 64;
constexpr int res_blocks(bool newton) { return newton ? 2 : 3; }  // resident blocks per SM (registers)

// Blocks of the tile kernel: a unit is one layer of a tile of tx x ty columns, a segment's
// units are numbered tile by tile, upward within a tile, and its nb blocks take equal
// contiguous ranges of them.
struct ResPlan {
  bool tile;
  int ltx, tilesx, tilesy, units, nb;
};

// Phi_c's neighbour (or ghost) at (i, j, k): pressure and conductivity.  False outside the
// grid's cells and ghosts, and for the ghost of a no-flux face.
__device__ __forceinline__ bool res_slot(const GridP& g, const SoilP& so, const BCP& bc, int i, int j, int k,
                                         const double* __restrict__ p, const double* __restrict__ ks, double& pv,
                                         double& kv) {
  const bool ox = (unsigned)i >= (unsigned)g.nx, oy = (unsigned)j >= (unsigned)g.ny;
  if (ox || oy) {
    if ((ox && oy) || i > g.nx || j > g.ny) return false;
    const int f = ox ? (i < 0 ? 0 : 1) : (j < 0 ? 2 : 3);
    if (bc.kind[f] == RICH_BC_NOFLUX) return false;
    const int ci = ox ? (i < 0 ? 0 : g.nx - 1) : i, cj = oy ? (j < 0 ? 0 : g.ny - 1) : j;
    pv = bc_value(bc, f, ci, cj, k, g.nx, g.ny);
    double kk = so.ks;
    if (bc.kind[f] == RICH_BC_INTERFACE) {  // a cell of the neighbouring subdomain, with its own K_s
      if (bc.gks[f]) kk = bc.gks[f][face_index(f, ci, cj, k, g.nx, g.ny)];
    } else if (ks) {
      kk = ks[ci + (long long)g.nx * (cj + (long long)g.ny * k)];
    }
    kv = conductivity_only(pv, kk, so);
    return true;
  }
  const long long c = i + (long long)g.nx * (j + (long long)g.ny * k);
  pv = p[c];
  const double kk = ks ? ks[c] : so.ks;
  kv = conductivity_only(pv, kk, ks ? kk * so.a : so.cka, so);
  return true;
}

// The layer below (side 0) or above (side 1) cell (i, j, k), kl its layer in its problem.
__device__ __forceinline__ bool res_vertical(const GridP& g, const SoilP& so, const BCP& bc, int i, int j, int k,
                                             int kl, int side, const double* __restrict__ p,
                                             const double* __restrict__ ks, double& pv, double& kv) {
  if (side ? kl < g.nzs - 1 : kl > 0) return res_slot(g, so, bc, i, j, side ? k + 1 : k - 1, p, ks, pv, kv);
  const int f = 4 + side;
  if (bc.kind[f] == RICH_BC_NOFLUX) return false;
  pv = bc_value(bc, f, i, j, k, g.nx, g.ny);
  double kk = so.ks;
  if (bc.kind[f] == RICH_BC_INTERFACE) {
    if (bc.gks[f]) kk = bc.gks[f][face_index(f, i, j, k, g.nx, g.ny)];
  } else if (ks) {
    kk = ks[i + (long long)g.nx * (j + (long long)g.ny * k)];
  }
  kv = conductivity_only(pv, kk, so);
  return true;
}

// K_av / h^2 of a face (KM = 0..3: that mean on every axis; 4: kmean's mean of this axis);
// dp = p_L - p_U.
template <int KM>
__device__ __forceinline__ double face_coef(int kmean, int axis, const GridP& g, double kL, double kU, double dp) {
  const int km = KM < 4 ? KM : axis_mean(kmean, axis);
  if (km == RICH_KMEAN_ARITH) return (kL + kU) * g.half_h2[axis];
  if (km == RICH_KMEAN_UPSTREAM) return (dp_upstream(dp) ? kU : kL) * g.inv_h2[axis];
  if (km == RICH_KMEAN_GEOMETRIC) return sqrt(kL * kU) * g.inv_h2[axis];
  const double s = kL + kU;
  return s > 0.0 ? (kL * kU) * (g.twice_h2[axis] * safe_rcp(s)) : 0.0;
}

// A cell's sum while its faces are added.
struct ResSum {
  double phi, mag;
};

// Horizontal face between the cell (pc, kc) and its neighbour on side `hi`.
template <int KM, bool MAG>
__device__ __forceinline__ void res_face(int kmean, int axis, bool hi, const GridP& g, double pc, double kc, double pn,
                                         double kn, ResSum& s) {
  const double dp = hi ? pc - pn : pn - pc;  // lower minus upper
  const double w = hi ? face_coef<KM>(kmean, axis, g, kc, kn, dp) : face_coef<KM>(kmean, axis, g, kn, kc, dp);
  s.phi = hi ? fma(w, dp, s.phi) : fma(-w, dp, s.phi);
  if (MAG) s.mag = fma(w, fabs(pc) + fabs(pn), s.mag);
}

// Vertical face, lower cell (pL, kL) to upper (pU, kU): flux out of the lower cell with the
// gravity term -(K_L + K_U) / (2 h_z), and the magnitude of its products.
template <int KM, bool MAG>
__device__ __forceinline__ void res_vface(int kmean, const GridP& g, double pL, double kL, double pU, double kU,
                                          double& t, double& m) {
  const double dp = pL - pU, ks = kL + kU;
  const double w = face_coef<KM>(kmean, 2, g, kL, kU, dp);
  t = fma(-g.half_hz, ks, w * dp);
  if (MAG) m = fma(w, fabs(pL) + fabs(pU), ks * g.half_hz);
}

// Storage term, and what Newton's form keeps for the Jacobian.  s_old NULL: s(p) itself,
// written to s_init.
template <bool NEWTON>
__device__ __forceinline__ void res_storage(const SoilP& so, long long c, double pc, const double* __restrict__ ks,
                                            const double* __restrict__ s_old, double rdt, double* __restrict__ K,
                                            double* __restrict__ dK, double* __restrict__ dS,
                                            double* __restrict__ s_init, ResSum& s) {
  double sc;
  if (NEWTON) {
    double ds, kc, dk;
    constit(pc, ks ? ks[c] : so.ks, so, sc, ds, kc, dk);
    K[c] = kc;
    dK[c] = dk;
    dS[c] = ds;
  } else {
    sc = saturation_only(pc, so);
  }
  double o;
  if (NEWTON && s_init) {
    o = sc;
    s_init[c] = sc;
  } else {
    o = s_old[c];
  }
  s.phi = (sc - o) * rdt;
  if (NEWTON) s.mag = (fabs(sc) + fabs(o)) * rdt;
}

// Sums of a block (N = blockDim.x threads) in a fixed order, and the largest |Phi| by its
// bits (a NaN's are above infinity's): results in thread 0.
template <int N, bool MAG>
__device__ __forceinline__ void res_block(double& a, double& m, unsigned long long& b) {
  __shared__ double sa[N / 32], sm[N / 32];
  __shared__ unsigned long long sb[N / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    if (MAG) m += __shfl_down_sync(0xffffffffu, m, o);
    const unsigned long long t = __shfl_down_sync(0xffffffffu, b, o);
    b = t > b ? t : b;
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) {
    sa[w] = a;
    if (MAG) sm[w] = m;
    sb[w] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < N / 32; ++q) {
      a += sa[q];
      if (MAG) m += sm[q];
      b = sb[q] > b ? sb[q] : b;
    }
  }
}

// Where the block sums go: quantity q of segment s, block b at part[q * stride + s * nb + b].
// ticket (one counter per segment, zero between launches), if not NULL: the segment's last
// block adds its partials up, in block order, into dst[q * nseg + s] and the pinned mirror,
// which takes the place of three single-block launches and a copy.
struct ResOut {
  double* part;
  long long stride;
  unsigned* ticket;
  double* dst;
  double* mirror;
};

template <int N, bool MAG>
__device__ __forceinline__ void res_finish(const ResOut& o, double a, double m, unsigned long long b) {
  const int nb = gridDim.x, seg = blockIdx.y, nseg = gridDim.y;
  res_block<N, MAG>(a, m, b);
  double* part = o.part + (long long)seg * nb;
  __shared__ bool last;
  if (threadIdx.x == 0) {
    part[blockIdx.x] = a;
    part[o.stride + blockIdx.x] = __longlong_as_double((long long)b);
    if (MAG) part[2 * o.stride + blockIdx.x] = m;
    last = false;
    if (o.ticket) {
      __threadfence();
      last = atomicAdd(&o.ticket[seg], 1u) == (unsigned)nb - 1;
    }
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  a = m = 0.0;
  b = 0;
  for (int t = threadIdx.x; t < nb; t += N) {
    a += __ldcg(&part[t]);
    const unsigned long long x = (unsigned long long)__double_as_longlong(__ldcg(&part[o.stride + t]));
    b = x > b ? x : b;
    if (MAG) m += __ldcg(&part[2 * o.stride + t]);
  }
  res_block<N, MAG>(a, m, b);
  if (threadIdx.x == 0) {
    const double r[3] = {a, __longlong_as_double((long long)b), m};
    for (int q = 0; q < (MAG ? 3 : 2); ++q) o.dst[q * nseg + seg] = o.mirror[q * nseg + seg] = r[q];
    o.ticket[seg] = 0;
  }
}

// Tile variant: tx x ty columns per block, marched upward.  Per layer a thread evaluates K
// of its own cell one layer ahead (in registers, for the vertical face), the block's halo
// ring is added in shared memory, and one barrier (double buffer) separates the layers.
template <int KM, bool NEWTON>
__global__ void __launch_bounds__(kResThreads, res_blocks(NEWTON)) k_residual_tile(
    GridP g, SoilP so, BCP bc, int kmean, ResPlan pl, const double* __restrict__ p, const double* __restrict__ s_old,
    const double* __restrict__ ks, double rdt, double* __restrict__ F, double* __restrict__ K, double* __restrict__ dK,
    double* __restrict__ dS, double* __restrict__ s_init, ResOut out) {
  __shared__ double sp[2][kResHalo], sk[2][kResHalo];
  const int tx = 1 << pl.ltx, ty = kResThreads >> pl.ltx, sx = tx + 2;
  const int lx = threadIdx.x & (tx - 1), ly = threadIdx.x >> pl.ltx;
  const int slot = (ly + 1) * sx + lx + 1;
  const int layers = g.nz / (int)gridDim.y, kseg = blockIdx.y * layers;
  double acc = 0.0, accm = 0.0;
  unsigned long long amax = 0;
  int buf = 0;
  const int u1 = (int)((blockIdx.x + 1LL) * pl.units / gridDim.x);
  for (int u = (int)((long long)blockIdx.x * pl.units / gridDim.x), run; u < u1; u += run) {
    const int t = u / layers, ks0 = u - t * layers;
    const int tj = t / pl.tilesx, i0 = (t - tj * pl.tilesx) << pl.ltx, j0 = tj * ty;
    const int kl0 = ks0 % g.nzs, kz = kseg + ks0 - kl0;  // layer within its problem, the problem's first layer
    run = min(u1 - u, g.nzs - kl0);
    const int kl1 = kl0 + run;
    const int i = i0 + lx, j = j0 + ly;
    const bool in = i < g.nx && j < g.ny;
    const bool fx0 = i > 0 || bc.kind[0] != RICH_BC_NOFLUX, fx1 = i < g.nx - 1 || bc.kind[1] != RICH_BC_NOFLUX;
    const bool fy0 = j > 0 || bc.kind[2] != RICH_BC_NOFLUX, fy1 = j < g.ny - 1 || bc.kind[3] != RICH_BC_NOFLUX;
    double pc = 0.0, kc = 0.0, tb = 0.0, mb = 0.0;  // this layer's cell; the flux through its bottom face
    res_slot(g, so, bc, i, j, kz + kl0, p, ks, pc, kc);
    if (in) {
      double pb, kb;
      if (res_vertical(g, so, bc, i, j, kz + kl0, kl0, 0, p, ks, pb, kb))
        res_vface<KM, NEWTON>(kmean, g, pb, kb, pc, kc, tb, mb);
    }
    for (int kl = kl0; kl < kl1; ++kl, buf ^= 1) {
      const int k = kz + kl;
      sp[buf][slot] = pc;
      sk[buf][slot] = kc;
      for (int h = threadIdx.x; h < 2 * (tx + ty); h += kResThreads) {  // the ring, corners left out
        const int q = h < 2 * ty ? h >> 1 : (h - 2 * ty) >> 1;
        const int hx = h < 2 * ty ? (h & 1 ? tx + 1 : 0) : q + 1, hy = h < 2 * ty ? q + 1 : (h & 1 ? ty + 1 : 0);
        double a = 0.0, b = 0.0;
        res_slot(g, so, bc, i0 + hx - 1, j0 + hy - 1, k, p, ks, a, b);
        sp[buf][hy * sx + hx] = a;
        sk[buf][hy * sx + hx] = b;
      }
      double pn = 0.0, kn = 0.0, tt = 0.0, mt = 0.0;
      bool up = false;
      if (in) {
        up = res_vertical(g, so, bc, i, j, k, kl, 1, p, ks, pn, kn);
        if (up) res_vface<KM, NEWTON>(kmean, g, pc, kc, pn, kn, tt, mt);
      } else if (kl + 1 < kl1) {  // a ghost slot of the next layer
        res_slot(g, so, bc, i, j, k + 1, p, ks, pn, kn);
      }
      __syncthreads();
      if (in) {
        const long long c = i + (long long)g.nx * (j + (long long)g.ny * k);
        ResSum s{0.0, 0.0};
        res_storage<NEWTON>(so, c, pc, ks, s_old, rdt, K, dK, dS, s_init, s);
        const double *a = sp[buf] + slot, *b = sk[buf] + slot;
        if (fx0) res_face<KM, NEWTON>(kmean, 0, false, g, pc, kc, a[-1], b[-1], s);
        if (fx1) res_face<KM, NEWTON>(kmean, 0, true, g, pc, kc, a[1], b[1], s);
        if (fy0) res_face<KM, NEWTON>(kmean, 1, false, g, pc, kc, a[-sx], b[-sx], s);
        if (fy1) res_face<KM, NEWTON>(kmean, 1, true, g, pc, kc, a[sx], b[sx], s);
        const double phi = (s.phi - tb) + tt;
        F[c] = phi;
        acc = fma(phi, phi, acc);
        if (NEWTON) {
          const double mag = (s.mag + mb) + mt;
          accm = fma(mag, mag, accm);
        }
        const unsigned long long ab = (unsigned long long)__double_as_longlong(phi) & 0x7fffffffffffffffull;
        amax = ab > amax ? ab : amax;
      }
      pc = pn;
      kc = kn;
      tb = tt;
      mb = mt;
    }
  }
  if (out.part) res_finish<kResThreads, NEWTON>(out, acc, accm, amax);
}

// Cell variant, for small grids and thin ones (planes that fill no tile): one cell per
// thread in small blocks, its neighbours' K recomputed, no barrier.
template <int KM, bool NEWTON>
__global__ void __launch_bounds__(kCellThreads) k_residual_cell(
    GridP g, SoilP so, BCP bc, int kmean, const double* __restrict__ p, const double* __restrict__ s_old,
    const double* __restrict__ ks, double rdt, double* __restrict__ F, double* __restrict__ K, double* __restrict__ dK,
    double* __restrict__ dS, double* __restrict__ s_init, ResOut out) {
  const long long ns = g.n / gridDim.y, c0 = blockIdx.y * ns;
  double acc = 0.0, accm = 0.0;
  unsigned long long amax = 0;
  for (long long c = c0 + blockIdx.x * (long long)kCellThreads + threadIdx.x; c < c0 + ns;
       c += (long long)gridDim.x * kCellThreads) {
    const int cc = (int)c, r = cc / g.nx;  // n is below 2^31
    const int i = cc - r * g.nx, k = r / g.ny, j = r - k * g.ny, kl = k % g.nzs;
    double pc, kc, pn, kn, tb = 0.0, mb = 0.0, tt = 0.0, mt = 0.0;
    res_slot(g, so, bc, i, j, k, p, ks, pc, kc);
    ResSum s{0.0, 0.0};
    res_storage<NEWTON>(so, c, pc, ks, s_old, rdt, K, dK, dS, s_init, s);
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const int d = f & 1 ? 1 : -1;
      if (res_slot(g, so, bc, f < 2 ? i + d : i, f < 2 ? j : j + d, k, p, ks, pn, kn))
        res_face<KM, NEWTON>(kmean, f >> 1, f & 1, g, pc, kc, pn, kn, s);
    }
    if (res_vertical(g, so, bc, i, j, k, kl, 0, p, ks, pn, kn))
      res_vface<KM, NEWTON>(kmean, g, pn, kn, pc, kc, tb, mb);
    if (res_vertical(g, so, bc, i, j, k, kl, 1, p, ks, pn, kn))
      res_vface<KM, NEWTON>(kmean, g, pc, kc, pn, kn, tt, mt);
    const double phi = (s.phi - tb) + tt;
    F[c] = phi;
    acc = fma(phi, phi, acc);
    if (NEWTON) {
      const double mag = (s.mag + mb) + mt;
      accm = fma(mag, mag, accm);
    }
    const unsigned long long ab = (unsigned long long)__double_as_longlong(phi) & 0x7fffffffffffffffull;
    amax = ab > amax ? ab : amax;
  }
  if (out.part) res_finish<kCellThreads, NEWTON>(out, acc, accm, amax);
}

// Which variant, and its shape.  The tile's width is the power of two (8 or more: 64-byte
// rows) with the fewest warps at work: those of a tile whose rows lie outside the grid
// skip the arithmetic, and a warp of the halo ring costs an eighth of a cell warp (its law
// against the law and the faces).  The ranges of units fill the SMs an integral number of
// times whether two (Newton's form) or three blocks are resident, so that both forms take the
// same sums; items of 8 layers left the fullest SM 20 % above the mean.  Each start of a column
// costs a law and a face more per thread, 5 % at 9 units per block.  Below kCellLimit cells
// there are too few tiles to fill the SMs, and a plane that leaves three quarters of its tiles
// empty wastes more than the cell variant's recomputed K.
constexpr long long kCellLimit = 40000;
inline ResPlan residual_plan(const GridP& g, int nseg, int max_blocks) {
  ResPlan pl{};
  double best = 1e300;
  for (int l = 3; l <= 8; ++l) {
    const int tx = 1 << l, ty = kResThreads >> l;
    const long long a = (g.nx + tx - 1) / tx, b = (g.ny + ty - 1) / ty;
    const int rows = tx < 32 ? 32 / tx : 1;  // grid rows under one warp
    const double cells = tx < 32 ? (double)a * ((g.ny + rows - 1) / rows) : (double)((g.nx + 31) / 32) * g.ny;
    const double cost = cells + 0.125 * a * b * ((2 * (tx + ty) + 31) / 32);
    if (cost < best) {
      best = cost;
      pl.ltx = l;
      pl.tilesx = (int)a;
      pl.tilesy = (int)b;
    }
  }
  const long long plane = (long long)pl.tilesx * pl.tilesy;
  pl.tile = g.n >= kCellLimit && 4LL * g.nx * g.ny >= plane * kResThreads;
  if (!pl.tile) {
    const long long nb = (g.n / nseg + kCellThreads - 1) / kCellThreads;
    pl.nb = (int)(nb < max_blocks ? nb : max_blocks);
    return pl;
  }
  pl.units = (int)(plane * (g.nz / nseg));  // at most n / 64: within int
  int nb = 6 * kNumSM / nseg;
  if (nb > max_blocks) nb = max_blocks;
  pl.nb = nb < 1 ? 1 : nb < pl.units ? nb : pl.units;
  return pl;
}

template <int KM, bool NEWTON>
static void residual_launch_km(const ResPlan& pl, int nseg, cudaStream_t st, const GridP& g, const SoilP& so,
                               const BCP& bc, int kmean, const double* p, const double* s_old, const double* ks,
                               double rdt, double* F, double* K, double* dK, double* dS, double* s_init,
                               const ResOut& out) {
  const dim3 grid(pl.nb, nseg);
  if (pl.tile)
    k_residual_tile<KM, NEWTON><<<grid, kResThreads, 0, st>>>(g, so, bc, kmean, pl, p, s_old, ks, rdt, F, K, dK, dS,
                                                              s_init, out);
  else
    k_residual_cell<KM, NEWTON><<<grid, kCellThreads, 0, st>>>(g, so, bc, kmean, p, s_old, ks, rdt, F, K, dK, dS,
                                                               s_init, out);
}

template <bool NEWTON>
static void residual_launch(const ResPlan& pl, int nseg, cudaStream_t st, const GridP& g, const SoilP& so,
                            const BCP& bc, int kmean, const double* p, const double* s_old, const double* ks,
                            double rdt, double* F, double* K, double* dK, double* dS, double* s_init, const ResOut& out) {
  switch (kmean) {
    case RICH_KMEAN_ARITH:
      return residual_launch_km<0, NEWTON>(pl, nseg, st, g, so, bc, kmean, p, s_old, ks, rdt, F, K, dK, dS, s_init, out);
    case RICH_KMEAN_UPSTREAM:
      return residual_launch_km<1, NEWTON>(pl, nseg, st, g, so, bc, kmean, p, s_old, ks, rdt, F, K, dK, dS, s_init, out);
    case RICH_KMEAN_HARMONIC:
      return residual_launch_km<2, NEWTON>(pl, nseg, st, g, so, bc, kmean, p, s_old, ks, rdt, F, K, dK, dS, s_init, out);
    case RICH_KMEAN_GEOMETRIC:
      return residual_launch_km<3, NEWTON>(pl, nseg, st, g, so, bc, kmean, p, s_old, ks, rdt, F, K, dK, dS, s_init, out);
    default:
      return residual_launch_km<4, NEWTON>(pl, nseg, st, g, so, bc, kmean, p, s_old, ks, rdt, F, K, dK, dS, s_init, out);
  }
}

}  // namespace rich

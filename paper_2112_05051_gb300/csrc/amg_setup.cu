// Smoothed-aggregation AMG setup on the GPU (Sec. 5.2: DSVMB-style decoupled
// smoothed aggregation; on one GPU the whole domain is one block).
//
//   strength   j != i strong iff max(a_ij^2, a_ji^2) >= theta_l^2 |a_ii a_jj|
//              (symmetrised; a_ji found by binary search, the pattern is symmetric),
//              theta_l = theta 2^-l on level l
//              (a constant threshold lets the coarse-operator density explode)
//   MIS-2      synchronous rounds over 64-bit tuples (state << 62 | key),
//              key(i) = top30(splitmix64(seed ^ i)) << 32 | i; two 1-hop max passes
//   aggregates roots numbered by an exclusive scan; pass 1 joins the strong
//              root neighbour of largest key, pass 2 the pass-1 neighbour whose
//              root has the largest key
//   P          (I - omega D^-1 A) P_tent, omega = 4/(3 max_i sum_j|a_ij|/|a_ii|)
//   Galerkin   A_c = R (A P), R = P^T
// Sparse products are row-wise expand-sort-compress: one warp per output row
// sorts 64-bit keys (column << 32 | product index) with a bitonic network and
// sums each column's products in product order, so patterns are structural
// and values deterministic.  The numeric refresh recomputes values on the kept
// patterns with one thread per row in the same product order.
#include <math_constants.h>

#include <algorithm>

#include "common.cuh"
#include "plist_limit.h"

namespace rich {

// ---------------------------------------------------------------- priorities

__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__device__ __forceinline__ uint64_t prio_key(uint64_t seed, long long i) {
  uint64_t pi = splitmix64(seed ^ (uint64_t)i);
  return ((pi >> 34) << 32) | (uint64_t)i;
}

constexpr uint64_t kStateShift = 62;
constexpr uint64_t kUndecided = 1;
constexpr uint64_t kIn = 2;
constexpr uint64_t kLow32 = 0xFFFFFFFFull;
constexpr uint64_t kKeyMask = (1ull << 62) - 1;

// ---------------------------------------------------------------- small kernels

__global__ void k_diag(int n, const int* __restrict__ rp, const int* __restrict__ col, const double* __restrict__ val,
                       double* __restrict__ d) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double v = 0.0;
    for (int e = rp[i]; e < rp[i + 1]; ++e)
      if (col[e] == i) v = val[e];
    d[i] = v;
  }
}

__device__ __forceinline__ int find_col(const int* __restrict__ col, int lo, int hi, int key) {
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (col[mid] < key) lo = mid + 1; else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ bool strong_sym(int i, int e, const int* __restrict__ rp, const int* __restrict__ col,
                                           const double* __restrict__ val, const double* __restrict__ d,
                                           double theta2) {
  int j = col[e];
  if (j == i) return false;
  double rhs = theta2 * fabs(d[i] * d[j]);
  double a = val[e];
  if (a * a >= rhs) return true;
  int q = find_col(col, rp[j], rp[j + 1], i);
  if (q < rp[j + 1] && col[q] == i) {
    double b = val[q];
    if (b * b >= theta2 * fabs(d[j] * d[i])) return true;
  }
  return false;
}

__global__ void k_strength(int n, const int* __restrict__ rp, const int* __restrict__ col,
                           const double* __restrict__ val, const double* __restrict__ d, double theta2,
                           const int* __restrict__ srp, int* __restrict__ cnt, int* __restrict__ scol) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int o = srp ? srp[i] : 0;
    int c = 0;
    for (int e = rp[i]; e < rp[i + 1]; ++e) {
      if (strong_sym(i, e, rp, col, val, d, theta2)) {
        if (scol) scol[o + c] = col[e];
        ++c;
      }
    }
    if (cnt) cnt[i] = c;
  }
}

// The same with a warp per row, for rows of more than a few entries (a thread per row walks
// 100 entries, each with a search in another row, one after another: 590 us for 1400 rows).
__global__ void k_strength_warp(int n, const int* __restrict__ rp, const int* __restrict__ col,
                                const double* __restrict__ val, const double* __restrict__ d, double theta2,
                                const int* __restrict__ srp, int* __restrict__ cnt, int* __restrict__ scol) {
  const int lane = threadIdx.x & 31;
  for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += (gridDim.x * blockDim.x) >> 5) {
    const int o = srp ? srp[i] : 0, e1 = rp[i + 1];
    int c = 0;
    for (int e0 = rp[i]; e0 < e1; e0 += 32) {
      const int e = e0 + lane;
      const bool s = e < e1 && strong_sym(i, e, rp, col, val, d, theta2);
      const unsigned m = __ballot_sync(0xffffffffu, s);
      if (s && scol) scol[o + c + __popc(m & ((1u << lane) - 1))] = col[e];
      c += __popc(m);
    }
    if (cnt && lane == 0) cnt[i] = c;
  }
}

static int strength(rich_ctx* c, const Csr<double>& A, const double* d, double theta2, const int* srp, int* cnt,
                    int* scol) {
  const int n = A.nrows;
  if (A.nnz > 12LL * n)
    k_strength_warp<<<grid_for(32LL * n), kBlock, 0, c->st>>>(n, A.rowptr, A.col, A.val, d, theta2, srp, cnt, scol);
  else
    k_strength<<<grid_for(n), kBlock, 0, c->st>>>(n, A.rowptr, A.col, A.val, d, theta2, srp, cnt, scol);
  RICH_LAUNCH_CHECK();
  return RICH_OK;
}

// Isolated nodes (no strong neighbour) start OUT: they join no aggregate.
__global__ void k_mis_init(int n, uint64_t seed, const int* __restrict__ srp, uint64_t* __restrict__ t) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    bool isolated = srp[i + 1] == srp[i];
    t[i] = (isolated ? 0ull : (kUndecided << kStateShift)) | prio_key(seed, i);
  }
}

// m[i] = max of v over the closed strength neighbourhood of i
__global__ void k_max_closed(int n, const int* __restrict__ srp, const int* __restrict__ scol,
                             const uint64_t* __restrict__ v, uint64_t* __restrict__ m) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    uint64_t best = v[i];
    for (int e = srp[i]; e < srp[i + 1]; ++e) {
      uint64_t w = v[scol[e]];
      best = w > best ? w : best;
    }
    m[i] = best;
  }
}

// second 1-hop pass and the state update of one MIS-2 round
__global__ void k_mis_update(int n, const int* __restrict__ srp, const int* __restrict__ scol,
                             const uint64_t* __restrict__ m1, uint64_t* __restrict__ t, int* __restrict__ undecided) {
  int any = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    uint64_t ti = t[i];
    if ((ti >> kStateShift) != kUndecided) continue;
    uint64_t best = m1[i];
    for (int e = srp[i]; e < srp[i + 1]; ++e) {
      uint64_t w = m1[scol[e]];
      best = w > best ? w : best;
    }
    if (best == ti) {
      t[i] = (kIn << kStateShift) | (ti & kKeyMask);
    } else if ((best >> kStateShift) == kIn) {
      t[i] = ti & kKeyMask;  // OUT = 0
    } else {
      any = 1;
    }
  }
  if (any) atomicOr(undecided, 1);
}

__global__ void k_is_root(int n, const uint64_t* __restrict__ t, int* __restrict__ isroot) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    isroot[i] = (t[i] >> kStateShift) == kIn ? 1 : 0;
}

__global__ void k_rootval(int n, const uint64_t* __restrict__ t, uint64_t* __restrict__ rv) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    uint64_t ti = t[i];
    rv[i] = (ti >> kStateShift) == kIn ? (ti & kKeyMask) + 1 : 0;
  }
}

// pass 1 result: agg (or -1) and the root index of pass-1 nodes (-1 otherwise)
__global__ void k_agg_pass1(int n, const uint64_t* __restrict__ t, const uint64_t* __restrict__ best,
                            const int* __restrict__ aggid, int* __restrict__ agg, int* __restrict__ p1root) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    bool root = (t[i] >> kStateShift) == kIn;
    p1root[i] = -1;
    if (root) {
      agg[i] = aggid[i];
    } else if (best[i] > 0) {
      int r = (int)((best[i] - 1) & kLow32);
      agg[i] = aggid[r];
      p1root[i] = r;
    } else {
      agg[i] = -1;
    }
  }
}

__global__ void k_val2(int n, const uint64_t* __restrict__ t, const int* __restrict__ p1root, uint64_t* __restrict__ v) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int r = p1root[i];
    v[i] = r >= 0 ? (t[r] & kKeyMask) + 1 : 0;
  }
}

__global__ void k_agg_pass2(int n, const int* __restrict__ srp, const uint64_t* __restrict__ best2,
                            const int* __restrict__ aggid, int* __restrict__ agg, int* __restrict__ unassigned) {
  int miss = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    if (agg[i] >= 0) continue;
    if (best2[i] > 0) agg[i] = aggid[(int)((best2[i] - 1) & kLow32)];
    else if (srp[i + 1] != srp[i]) miss = 1;  // isolated nodes stay unaggregated (agg = -1)
  }
  if (miss) atomicOr(unassigned, 1);
}

// Pass 3: a node left out by passes 1-2 (no strong neighbour) whose row is not
// diagonally dominant (a_ii < 2 sum_{j!=i} |a_ij|) joins the aggregate of its
// aggregated neighbour j with the largest (fp32 |a_ij|, key(j)).  On high-contrast
// fields such a row sums to about zero although every coupling is weak relative to
// the neighbours' diagonals; left out, its error is corrected by the smoother alone.
// Reads the aggregates of passes 1-2 (agg_in) only, so the pass is synchronous.
__global__ void k_agg_pass3(int n, const int* __restrict__ rp, const int* __restrict__ col,
                            const double* __restrict__ val, uint64_t seed, const int* __restrict__ agg_in,
                            int* __restrict__ agg_out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int a = agg_in[i];
    if (a >= 0) continue;
    double diag = 0.0, off = 0.0;
    for (int e = rp[i]; e < rp[i + 1]; ++e) {
      if (col[e] == i) diag = val[e];
      else off += fabs(val[e]);
    }
    if (!(fabs(diag) < 2.0 * off)) continue;
    int bj = -1;
    float bw = 0.0f;
    uint64_t bk = 0;
    for (int e = rp[i]; e < rp[i + 1]; ++e) {
      int j = col[e];
      if (j == i || agg_in[j] < 0) continue;
      float w = (float)fabs(val[e]);
      uint64_t kj = prio_key(seed, j);
      if (bj < 0 || w > bw || (w == bw && kj > bk)) {
        bj = j;
        bw = w;
        bk = kj;
      }
    }
    if (bj >= 0) agg_out[i] = agg_in[bj];
  }
}

// P_tent: one unit entry per aggregated node, empty rows for isolated nodes
__global__ void k_ptent_count(int n, const int* __restrict__ agg, int* __restrict__ cnt) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) cnt[i] = agg[i] >= 0;
}
__global__ void k_ptent_fill(int n, const int* __restrict__ agg, const int* __restrict__ rp, int* __restrict__ col) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    if (agg[i] >= 0) col[rp[i]] = agg[i];
}

__global__ void k_rowratio(int n, const int* __restrict__ rp, const double* __restrict__ val,
                           const double* __restrict__ d, double* __restrict__ partials) {
  double m = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int e = rp[i]; e < rp[i + 1]; ++e) s += fabs(val[e]);
    double r = s / fabs(d[i]);
    m = (r > m || r != r) ? r : m;
  }
  m = block_max(m);
  if (threadIdx.x == 0) partials[blockIdx.x] = m;
}

// S = I - omega D^-1 A on the pattern of A (same operation order as the oracle)
__global__ void k_smoother_vals(int n, const int* __restrict__ rp, const int* __restrict__ col,
                                const double* __restrict__ val, const double* __restrict__ d, double omega,
                                double* __restrict__ sval) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    for (int e = rp[i]; e < rp[i + 1]; ++e) sval[e] = -omega * val[e] / d[i] + (col[e] == i ? 1.0 : 0.0);
}

__global__ void k_seq(int n, int* __restrict__ a) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += gridDim.x * blockDim.x) a[i] = i;
}

__global__ void k_fill(long long n, double v, double* __restrict__ a) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    a[i] = v;
}

__global__ void k_l1dinv(int n, const int* __restrict__ rp, const double* __restrict__ val, double* __restrict__ dinv,
                         float* __restrict__ dinv32) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int e = rp[i]; e < rp[i + 1]; ++e) s += fabs(val[e]);
    double r = 1.0 / s;
    dinv[i] = r;
    if (dinv32) dinv32[i] = (float)r;
  }
}

__global__ void k_l1dinv32(int n, const int* __restrict__ rp, const float* __restrict__ val, float* __restrict__ dinv32) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    float s = 0.0f;
    for (int e = rp[i]; e < rp[i + 1]; ++e) s += fabsf(val[e]);
    dinv32[i] = 1.0f / s;
  }
}

__global__ void k_cast(long long n, const double* __restrict__ a, float* __restrict__ b) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    b[i] = (float)a[i];
}

// ---------------------------------------------------------------- transpose

__global__ void k_tr_count(int n, const int* __restrict__ rp, const int* __restrict__ col, int* __restrict__ cnt) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    for (int e = rp[i]; e < rp[i + 1]; ++e) atomicAdd(&cnt[col[e]], 1);
}

__global__ void k_tr_fill(int n, const int* __restrict__ rp, const int* __restrict__ col,
                          const double* __restrict__ val, const int* __restrict__ trp, int* __restrict__ fillc,
                          int* __restrict__ tcol, double* __restrict__ tval) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    for (int e = rp[i]; e < rp[i + 1]; ++e) {
      int J = col[e];
      int pos = trp[J] + atomicAdd(&fillc[J], 1);
      tcol[pos] = i;
      tval[pos] = val[e];
    }
}

// ---------------------------------------------------------------- expand-sort-compress SpGEMM

__global__ void k_spgemm_upper(int n, const int* __restrict__ arp, const int* __restrict__ acol,
                               const int* __restrict__ brp, int* __restrict__ u) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    long long s = 0;
    for (int e = arp[i]; e < arp[i + 1]; ++e) s += brp[acol[e] + 1] - brp[acol[e]];
    u[i] = s > 2147483647LL ? 2147483647 : (int)s;
  }
}

__global__ void k_max_int(int n, const int* __restrict__ a, int* __restrict__ out) {
  int m = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) m = max(m, a[i]);
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

__device__ __forceinline__ void warp_bitonic_sort(uint64_t* keys, int M, int lane) {
  for (int k = 2; k <= M; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = lane; t < M; t += 32) {
        int ixj = t ^ j;
        if (ixj > t) {
          uint64_t a = keys[t], b = keys[ixj];
          bool asc = (t & k) == 0;
          if ((a > b) == asc) {
            keys[t] = b;
            keys[ixj] = a;
          }
        }
      }
      __syncwarp();
    }
  }
}

constexpr int kEscCap = 1024;    // most products per row the shared-memory ESC kernel takes

// mode 0: cnt[row] = number of distinct columns; mode 1: write the compressed row at crp[row];
// mode 2 (single pass): write it at the row's product offset uoff[row] of a temporary
// and set cnt[row].
// Each warp owns `cap` key/value slots of shared memory (cap = the launch's largest
// product count rounded up to a power of two, at most kEscCap), so short rows
// (the 7-point level: tens of products) run many warps per SM.  Rows whose product
// count exceeds kEscCap are left to k_spgemm_hash.
__global__ void k_spgemm_esc(int nrows, const int* __restrict__ arp, const int* __restrict__ acol,
                             const double* __restrict__ aval, const int* __restrict__ brp,
                             const int* __restrict__ bcol, const double* __restrict__ bval,
                             const int* __restrict__ u, int mode, const int* __restrict__ crp,
                             const long long* __restrict__ uoff, int* __restrict__ ccol, double* __restrict__ cval,
                             int* __restrict__ cnt, int cap) {
  extern __shared__ unsigned char smem[];
  int wpb = blockDim.x >> 5;
  int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint64_t* skeys = reinterpret_cast<uint64_t*>(smem) + (size_t)w * cap;
  double* svals = reinterpret_cast<double*>(smem + (size_t)wpb * cap * sizeof(uint64_t)) + (size_t)w * cap;
  for (int row = blockIdx.x * wpb + w; row < nrows; row += gridDim.x * wpb) {
    int ur = u[row];
    if (ur > cap) continue;
    uint64_t* keys = skeys;
    double* vals = svals;
    int M = 1;
    while (M < ur) M <<= 1;
    // expand in product order: A entries in column order, then B entries in column order
    int t0 = 0;
    for (int e = arp[row]; e < arp[row + 1]; ++e) {
      int j = acol[e];
      double a = aval ? aval[e] : 1.0;
      int b0 = brp[j], len = brp[j + 1] - b0;
      for (int q = lane; q < len; q += 32) {
        int t = t0 + q;
        keys[t] = ((uint64_t)(uint32_t)bcol[b0 + q] << 32) | (uint32_t)t;
        vals[t] = a * (bval ? bval[b0 + q] : 1.0);
      }
      t0 += len;
    }
    for (int t = ur + lane; t < M; t += 32) keys[t] = ~0ull;
    __syncwarp();
    warp_bitonic_sort(keys, M, lane);
    // segment heads
    const long long base = mode == 1 ? (long long)crp[row] : (mode == 2 ? uoff[row] : 0);
    int running = 0;
    for (int t0s = 0; t0s < ur; t0s += 32) {
      int t = t0s + lane;
      bool head = false;
      uint32_t c = 0;
      if (t < ur) {
        c = (uint32_t)(keys[t] >> 32);
        head = (t == 0) || ((uint32_t)(keys[t - 1] >> 32) != c);
      }
      unsigned mask = __ballot_sync(0xffffffffu, head);
      if (mode != 0 && head) {
        const long long pos = base + running + __popc(mask & ((1u << lane) - 1));
        double s = 0.0;
        for (int q = t; q < ur && (uint32_t)(keys[q] >> 32) == c; ++q) s += vals[(uint32_t)(keys[q] & kLow32)];
        ccol[pos] = (int)c;
        cval[pos] = s;
      }
      running += __popc(mask);
    }
    if (mode != 1 && lane == 0) cnt[row] = running;
    __syncwarp();
  }
}

// The same for products with fewer than 2^kSortCol columns: keys of 32 bits (column, product
// index), sorted in registers.  A lane holds K consecutive keys, so that the network's
// short distances are register exchanges and the long ones shuffles; the products of 32 A
// entries at a time are spread over the lanes through a scan of their B rows' lengths, so
// that the loads of a row are in flight together.  Sums, order and results are k_spgemm_esc's.
// 64^3, A_1 P_1 (29k rows, 210 products on average): 1480 us in shared memory with 64-bit
// keys, 16 kB per warp and one A entry after another.
constexpr int kSortCol = 22, kSortIdx = 32 - kSortCol;
static_assert((1 << kSortIdx) >= kEscCap, "a product index fits beside the column");

template <int K>
__device__ __forceinline__ void warp_sort_keys(unsigned* keys, int u, int lane) {
  unsigned a[K];
#pragma unroll
  for (int r = 0; r < K; ++r) a[r] = lane * K + r < u ? keys[lane * K + r] : 0xffffffffu;
#pragma unroll
  for (int k = 2; k <= 32 * K; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= K) {
        const bool keep_min = ((lane & (j / K)) == 0) == ((lane & (k / K)) == 0);
#pragma unroll
        for (int r = 0; r < K; ++r) {
          const unsigned o = __shfl_xor_sync(0xffffffffu, a[r], j / K);
          a[r] = keep_min ? min(a[r], o) : max(a[r], o);
        }
      } else {
#pragma unroll
        for (int r = 0; r < K; ++r)
          if ((r & j) == 0) {
            const bool asc = k < K ? (r & k) == 0 : (lane & (k / K)) == 0;
            const unsigned lo = min(a[r], a[r ^ j]), hi = max(a[r], a[r ^ j]);
            a[r] = asc ? lo : hi;
            a[r ^ j] = asc ? hi : lo;
          }
      }
    }
  }
  __syncwarp();
#pragma unroll
  for (int r = 0; r < K; ++r)
    if (lane * K + r < u) keys[lane * K + r] = a[r];
  __syncwarp();
}

// Rows with umin < products <= cap (cap slots of shared memory per warp), cap <= 32 KMAX.
// The kernel waits on loads, so the classes are compiled apart: registers for short keys
// only let twice the warps in (262k rows of 24 products: 340 us with all sizes in one).
template <int KMAX>
__global__ void __launch_bounds__(256, KMAX <= 2 ? 6 : KMAX <= 8 ? 5 : 2) k_spgemm_sort(int nrows, const int* __restrict__ arp,
                                                     const int* __restrict__ acol, const double* __restrict__ aval,
                                                     const int* __restrict__ brp, const int* __restrict__ bcol,
                                                     const double* __restrict__ bval, const int* __restrict__ u,
                                                     int mode, const int* __restrict__ crp,
                                                     const long long* __restrict__ uoff, int* __restrict__ ccol,
                                                     double* __restrict__ cval, int* __restrict__ cnt, int umin,
                                                     int cap) {
  extern __shared__ __align__(8) unsigned char smem[];
  __shared__ int pre_all[8][33], bst_all[8][32];
  __shared__ double av_all[8][32];
  const int wpb = blockDim.x >> 5, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double* vals = reinterpret_cast<double*>(smem) + (size_t)w * cap;
  unsigned* keys = reinterpret_cast<unsigned*>(smem + (size_t)wpb * cap * sizeof(double)) + (size_t)w * cap;
  int *pre = pre_all[w], *bst = bst_all[w];
  double* av = av_all[w];
  for (int row = blockIdx.x * wpb + w; row < nrows; row += gridDim.x * wpb) {
    const int ur = u[row];
    if (ur > cap || ur <= umin) {
      if (ur == 0 && umin == 0 && mode != 1 && lane == 0) cnt[row] = 0;
      continue;
    }
    // expand in product order: A entries in column order, then B entries in column order
    int t0 = 0;
    const int a1 = arp[row + 1];
    for (int e0 = arp[row]; e0 < a1; e0 += 32) {
      const int e = e0 + lane;
      const bool has = e < a1;
      const int j = has ? acol[e] : 0;
      const int b0 = has ? brp[j] : 0, len = has ? brp[j + 1] - b0 : 0;
      int inc = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
      }
      const int total = __shfl_sync(0xffffffffu, inc, 31);
      pre[lane + 1] = inc;
      if (lane == 0) pre[0] = 0;
      bst[lane] = b0;
      av[lane] = has && aval ? aval[e] : 1.0;
      __syncwarp();
      for (int p = lane; p < total; p += 32) {
        int lo = 0, hi = 32;  // owner q of product p: pre[q] <= p < pre[q+1]
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (pre[mid] <= p) lo = mid; else hi = mid;
        }
        const int f = bst[lo] + (p - pre[lo]);
        keys[t0 + p] = (unsigned)bcol[f] << kSortIdx | (unsigned)(t0 + p);
        vals[t0 + p] = av[lo] * (bval ? bval[f] : 1.0);
      }
      t0 += total;
      __syncwarp();
    }
    if (KMAX <= 2) {
      if (ur <= 32) warp_sort_keys<1>(keys, ur, lane);
      else warp_sort_keys<2>(keys, ur, lane);
    } else if (KMAX <= 8) {
      if (ur <= 128) warp_sort_keys<4>(keys, ur, lane);
      else warp_sort_keys<8>(keys, ur, lane);
    } else {
      if (ur <= 512) warp_sort_keys<16>(keys, ur, lane);
      else warp_sort_keys<32>(keys, ur, lane);
    }
    // segment heads
    const long long base = mode == 1 ? (long long)crp[row] : (mode == 2 ? uoff[row] : 0);
    int running = 0;
    for (int s0 = 0; s0 < ur; s0 += 32) {
      const int t = s0 + lane;
      const unsigned c = t < ur ? keys[t] >> kSortIdx : 0u;
      const bool head = t < ur && (t == 0 || keys[t - 1] >> kSortIdx != c);
      const unsigned mask = __ballot_sync(0xffffffffu, head);
      if (mode != 0 && head) {
        const long long pos = base + running + __popc(mask & ((1u << lane) - 1));
        double s = 0.0;
        for (int q = t; q < ur && keys[q] >> kSortIdx == c; ++q) s += vals[keys[q] & ((1u << kSortIdx) - 1)];
        ccol[pos] = (int)c;
        cval[pos] = s;
      }
      running += __popc(mask);
    }
    if (mode != 1 && lane == 0) cnt[row] = running;
    __syncwarp();
  }
}

// Rows with more than kEscCap products: one block per row accumulates the products
// into a shared-memory hash table keyed by column (linear probing, atomicCAS), then
// sorts the occupied keys.  The column set is exact; the FP64 sums depend on the
// order of the shared-memory atomics (rounding-level differences only).
constexpr int kHashSlots = 8192;
constexpr int kHashThreads = 256;

__global__ void __launch_bounds__(kHashThreads) k_spgemm_hash(
    int nrows, const int* __restrict__ arp, const int* __restrict__ acol, const double* __restrict__ aval,
    const int* __restrict__ brp, const int* __restrict__ bcol, const double* __restrict__ bval,
    const int* __restrict__ u, int mode, const int* __restrict__ crp, const long long* __restrict__ uoff,
    int* __restrict__ ccol, double* __restrict__ cval, int* __restrict__ cnt, int* __restrict__ overflow) {
  extern __shared__ unsigned char smem[];
  int* hkey = reinterpret_cast<int*>(smem);
  double* hval = reinterpret_cast<double*>(smem + kHashSlots * sizeof(int));
  __shared__ int nfill;
  __shared__ int fail;
  __shared__ int pre[kHashThreads + 1], bst[kHashThreads], wsum[kHashThreads / 32];
  __shared__ double av[kHashThreads];
  for (int row = blockIdx.x; row < nrows; row += gridDim.x) {
    if (u[row] <= kEscCap) continue;
    for (int t = threadIdx.x; t < kHashSlots; t += blockDim.x) {
      hkey[t] = -1;
      hval[t] = 0.0;
    }
    if (threadIdx.x == 0) {
      nfill = 0;
      fail = 0;
    }
    __syncthreads();
    // products of 256 A entries at a time, spread over the block through a scan of their B
    // rows' lengths (one A entry after another left most threads idle: 1270 us for 1400 rows)
    for (int e0 = arp[row]; e0 < arp[row + 1]; e0 += kHashThreads) {
      const int e = e0 + threadIdx.x;
      const bool has = e < arp[row + 1];
      const int j = has ? acol[e] : 0;
      const int b0 = has ? brp[j] : 0, len = has ? brp[j + 1] - b0 : 0;
      const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
      int inc = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
      }
      if (lane == 31) wsum[wid] = inc;
      bst[threadIdx.x] = b0;
      av[threadIdx.x] = has && aval ? aval[e] : 1.0;
      __syncthreads();
      int add = 0;
      for (int q = 0; q < wid; ++q) add += wsum[q];
      pre[threadIdx.x + 1] = inc + add;
      if (threadIdx.x == 0) pre[0] = 0;
      __syncthreads();
      const int total = pre[kHashThreads];
      for (int p = threadIdx.x; p < total; p += blockDim.x) {
        int lo = 0, hi = kHashThreads;
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (pre[mid] <= p) lo = mid; else hi = mid;
        }
        const int f = bst[lo] + (p - pre[lo]);
        int col = bcol[f];
        double v = av[lo] * (bval ? bval[f] : 1.0);
        unsigned h = ((unsigned)col * 2654435761u) & (kHashSlots - 1);
        int probes = 0;
        for (;;) {
          int k = ((volatile int*)hkey)[h];
          if (k == col) break;
          if (k == -1) {
            int prev = atomicCAS(&hkey[h], -1, col);
            if (prev == -1 || prev == col) break;
          }
          h = (h + 1) & (kHashSlots - 1);
          if (++probes >= kHashSlots) {
            fail = 1;
            break;
          }
        }
        if (probes < kHashSlots) atomicAdd(&hval[h], v);
      }
      __syncthreads();
    }
    if (fail) {
      if (threadIdx.x == 0) atomicOr(overflow, 1);
      __syncthreads();
      continue;
    }
    // compact occupied slots to the front: (col << 32 | slot) keys reuse hkey/hval storage order
    // via a second pass; collect into a sorted list with a block bitonic sort of 64-bit keys
    // stored in the (now free) upper part of smem.
    uint64_t* keys = reinterpret_cast<uint64_t*>(smem + kHashSlots * (sizeof(int) + sizeof(double)));
    for (int t = threadIdx.x; t < kHashSlots; t += blockDim.x) {
      int k = hkey[t];
      if (k >= 0) {
        int pos = atomicAdd(&nfill, 1);
        keys[pos] = ((uint64_t)(uint32_t)k << 32) | (uint32_t)t;
      }
    }
    __syncthreads();
    int L = nfill;
    int M = 1;
    while (M < L) M <<= 1;
    for (int t = L + threadIdx.x; t < M; t += blockDim.x) keys[t] = ~0ull;
    __syncthreads();
    for (int k = 2; k <= M; k <<= 1) {
      for (int jj = k >> 1; jj > 0; jj >>= 1) {
        for (int t = threadIdx.x; t < M; t += blockDim.x) {
          int ixj = t ^ jj;
          if (ixj > t) {
            uint64_t x = keys[t], y = keys[ixj];
            bool asc = (t & k) == 0;
            if ((x > y) == asc) {
              keys[t] = y;
              keys[ixj] = x;
            }
          }
        }
        __syncthreads();
      }
    }
    if (mode != 1 && threadIdx.x == 0) cnt[row] = L;
    if (mode != 0) {
      const long long base = mode == 1 ? (long long)crp[row] : uoff[row];
      for (int t = threadIdx.x; t < L; t += blockDim.x) {
        ccol[base + t] = (int)(keys[t] >> 32);
        cval[base + t] = hval[(uint32_t)(keys[t] & kLow32)];
      }
    }
    __syncthreads();
  }
}

// Values of C = A B on C's known pattern.  Rows with at most kNumSmall products:
// one thread per row, products in the ESC order (sums identical to the symbolic
// pass).  Larger rows: k_spgemm_numeric_block.
constexpr int kNumSmall = 64;

template <class T>
__global__ void k_spgemm_numeric(int nrows, const int* __restrict__ arp, const int* __restrict__ acol,
                                 const T* __restrict__ aval, const int* __restrict__ brp,
                                 const int* __restrict__ bcol, const T* __restrict__ bval,
                                 const int* __restrict__ crp, const int* __restrict__ ccol,
                                 T* __restrict__ cval, const int* __restrict__ u) {
  constexpr int kReg = 32;  // rows with at most kReg entries accumulate in a per-thread array
  for (int row = blockIdx.x * blockDim.x + threadIdx.x; row < nrows; row += gridDim.x * blockDim.x) {
    if (u[row] > kNumSmall) continue;
    int c0 = crp[row], c1 = crp[row + 1], L = c1 - c0;
    if (L <= kReg) {
      int cc[kReg];
      T acc[kReg];
#pragma unroll
      for (int q = 0; q < kReg; ++q) {
        cc[q] = q < L ? ccol[c0 + q] : -1;
        acc[q] = T(0);
      }
      for (int e = arp[row]; e < arp[row + 1]; ++e) {
        int j = acol[e];
        T a = aval[e];
        for (int f = brp[j]; f < brp[j + 1]; ++f) {
          int key = bcol[f];
          T v = a * bval[f];
          int pos = 0;
#pragma unroll
          for (int q = 0; q < kReg; ++q) pos = cc[q] == key ? q : pos;
          acc[pos] += v;
        }
      }
      for (int q = 0; q < L; ++q) cval[c0 + q] = acc[q];
      continue;
    }
    for (int q = c0; q < c1; ++q) cval[q] = T(0);
    for (int e = arp[row]; e < arp[row + 1]; ++e) {
      int j = acol[e];
      T a = aval[e];
      for (int f = brp[j]; f < brp[j + 1]; ++f) {
        int pos = find_col(ccol, c0, c1, bcol[f]);
        cval[pos] += a * bval[f];
      }
    }
  }
}

// One warp per row with more than kNumSmall products and at most kWarpL output
// entries: the row's columns and accumulators sit in the warp's slice of shared
// memory; A entries are taken 32 at a time, a warp scan of their B-row lengths
// flattens the products over the lanes.
constexpr int kWarpL = 256;
constexpr int kWarpRowsPerBlock = 8;

template <class T>
__global__ void __launch_bounds__(32 * kWarpRowsPerBlock) k_spgemm_numeric_warp(
    int nrows, const int* __restrict__ arp, const int* __restrict__ acol, const T* __restrict__ aval,
    const int* __restrict__ brp, const int* __restrict__ bcol, const T* __restrict__ bval,
    const int* __restrict__ crp, const int* __restrict__ ccol, T* __restrict__ cval,
    const int* __restrict__ u) {
  __shared__ T sacc_all[kWarpRowsPerBlock][kWarpL];
  __shared__ int scol_all[kWarpRowsPerBlock][kWarpL];
  __shared__ int pre_all[kWarpRowsPerBlock][33];
  __shared__ int bst_all[kWarpRowsPerBlock][32];
  __shared__ T av_all[kWarpRowsPerBlock][32];
  int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  T* sacc = sacc_all[w];
  int* scol = scol_all[w];
  int* pre = pre_all[w];
  int nw = gridDim.x * kWarpRowsPerBlock;
  for (int row = blockIdx.x * kWarpRowsPerBlock + w; row < nrows; row += nw) {
    int c0 = crp[row], c1 = crp[row + 1], L = c1 - c0;
    if (u[row] <= kNumSmall || L > kWarpL) continue;
    for (int t = lane; t < L; t += 32) {
      scol[t] = ccol[c0 + t];
      sacc[t] = T(0);
    }
    __syncwarp();
    for (int e0 = arp[row]; e0 < arp[row + 1]; e0 += 32) {
      int e = e0 + lane;
      bool has = e < arp[row + 1];
      int j = has ? acol[e] : 0;
      T a = has ? aval[e] : T(0);
      int b0 = has ? brp[j] : 0;
      int len = has ? brp[j + 1] - b0 : 0;
      int inc = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
      }
      pre[lane + 1] = inc;
      if (lane == 0) pre[0] = 0;
      int total = __shfl_sync(0xffffffffu, inc, 31);
      bst_all[w][lane] = b0;
      av_all[w][lane] = a;
      __syncwarp();
      for (int t = lane; t < total; t += 32) {
        int lo = 0, hi = 32;  // owner q of product t: pre[q] <= t < pre[q+1]
        while (hi - lo > 1) {
          int mid = (lo + hi) >> 1;
          if (pre[mid] <= t) lo = mid; else hi = mid;
        }
        int f = bst_all[w][lo] + (t - pre[lo]);
        int key = bcol[f];
        T v = av_all[w][lo] * bval[f];
        int pos = find_col(scol, 0, L, key);
        atomicAdd(&sacc[pos], v);
      }
      __syncwarp();
    }
    for (int t = lane; t < L; t += 32) cval[c0 + t] = sacc[t];
    __syncwarp();
  }
}

// One block per row with more than kNumSmall products.  The row's products are
// flattened: a block scan of the B-row lengths over the row's A entries gives
// each product index t an (A entry, B entry) pair, so every thread has work
// however short the B rows are.  The row's column list and accumulators sit in
// shared memory (rows up to kNumLmax entries; longer rows accumulate in global
// memory); products are added with atomics (rounding-level order dependence).
constexpr int kNumLmax = 4096;
constexpr int kNumAmax = 2048;   // A entries per row staged at once
constexpr int kNumThreads = 256;
constexpr int kDenseCols = 8192; // C with at most this many columns: accumulate by column directly

// DENSE: the shared accumulator is indexed by column (C has <= kDenseCols columns),
// so a product needs no search; otherwise the row's sorted column list is searched.
template <class T, bool DENSE>
__global__ void __launch_bounds__(kNumThreads) k_spgemm_numeric_block(
    int nrows, const int* __restrict__ arp, const int* __restrict__ acol, const T* __restrict__ aval,
    const int* __restrict__ brp, const int* __restrict__ bcol, const T* __restrict__ bval,
    const int* __restrict__ crp, const int* __restrict__ ccol, T* __restrict__ cval,
    const int* __restrict__ u, int ncols) {
  // dynamic shared memory: sacc[kNumLmax] av[kNumAmax] (doubles), then scol[kNumLmax]
  // off[kNumAmax + 1] bstart[kNumAmax] (ints)
  extern __shared__ unsigned char dsm[];
  T* sacc = reinterpret_cast<T*>(dsm);
  T* av = sacc + (DENSE ? kDenseCols : kNumLmax);
  int* scol = reinterpret_cast<int*>(av + kNumAmax);
  int* off = scol + kNumLmax;         // prefix of B-row lengths over the staged A entries
  int* bstart = off + kNumAmax + 1;
  __shared__ int wsum[kNumThreads / 32];
  for (int row = blockIdx.x; row < nrows; row += gridDim.x) {
    if (u[row] <= kNumSmall) continue;
    int c0 = crp[row], c1 = crp[row + 1], L = c1 - c0;
    if (L <= kWarpL) continue;  // k_spgemm_numeric_warp
    bool sh = DENSE || L <= kNumLmax;
    if (DENSE) {
      for (int t = threadIdx.x; t < L; t += blockDim.x) sacc[ccol[c0 + t]] = T(0);
    } else if (sh) {
      for (int t = threadIdx.x; t < L; t += blockDim.x) {
        scol[t] = ccol[c0 + t];
        sacc[t] = T(0);
      }
    } else {
      for (int t = threadIdx.x; t < L; t += blockDim.x) cval[c0 + t] = T(0);
    }
    __syncthreads();
    for (int e0 = arp[row]; e0 < arp[row + 1]; e0 += kNumAmax) {
      int na = min(kNumAmax, arp[row + 1] - e0);
      // stage A entries and the lengths of their B rows; block-wide exclusive scan
      int per = (na + blockDim.x - 1) / blockDim.x;
      int lo = threadIdx.x * per, hi = min(na, lo + per);
      int local = 0;
      for (int q = lo; q < hi; ++q) {
        int j = acol[e0 + q];
        int b0 = brp[j];
        bstart[q] = b0;
        av[q] = aval[e0 + q];
        int len = brp[j + 1] - b0;
        off[q] = local;
        local += len;
      }
      // exclusive scan of the per-thread totals
      int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
      int inc = local;
      for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
      }
      if (lane == 31) wsum[wid] = inc;
      __syncthreads();
      int wbase = 0;
      for (int q = 0; q < wid; ++q) wbase += wsum[q];
      int tbase = wbase + inc - local;
      for (int q = lo; q < hi; ++q) off[q] += tbase;
      __syncthreads();
      int total = 0;
      for (int q = 0; q < (int)(blockDim.x >> 5); ++q) total += wsum[q];
      if (threadIdx.x == 0) off[na] = total;
      __syncthreads();
      for (int t = threadIdx.x; t < total; t += blockDim.x) {
        // A entry q with off[q] <= t < off[q+1]
        int lo2 = 0, hi2 = na;
        while (hi2 - lo2 > 1) {
          int mid = (lo2 + hi2) >> 1;
          if (off[mid] <= t) lo2 = mid; else hi2 = mid;
        }
        int f = bstart[lo2] + (t - off[lo2]);
        int key = bcol[f];
        T v = av[lo2] * bval[f];
        if (DENSE) {
          atomicAdd(&sacc[key], v);
        } else if (sh) {
          int pos = find_col(scol, 0, L, key);
          atomicAdd(&sacc[pos], v);
        } else {
          int pos = find_col(ccol, c0, c1, key);
          atomicAdd(&cval[pos], v);
        }
      }
      __syncthreads();
    }
    if (DENSE)
      for (int t = threadIdx.x; t < L; t += blockDim.x) cval[c0 + t] = sacc[ccol[c0 + t]];
    else if (sh)
      for (int t = threadIdx.x; t < L; t += blockDim.x) cval[c0 + t] = sacc[t];
    __syncthreads();
  }
}

// ---------------------------------------------------------------- Galerkin refresh by product lists
// The patterns of A P and R (A P) do not change between refreshes, so the pair
// (A entry, B entry) behind each scalar product, and the C entry it adds to, are
// the same every time.  k_plist enumerates the products of each row (one warp
// per row, A entries 32 at a time, a warp scan of their B-row lengths spreads
// the products over the lanes) and either counts the products of every C entry
// or files each pair into its C entry's slots (ProdList), which k_pl_shape lays out from
// the counts; k_pl_sort or k_pl_rank then orders each entry's pairs by A entry, which is
// the order a row-by-row product sums in.
constexpr int kPlWarps = 8;
constexpr int kPlCols = 512;  // columns of a C row searched in shared memory

// WIDE: a block per row (rows of thousands of products), its warps taking the row's A
// entries in turn; the order within a segment is settled by k_pl_rank either way.
template <bool FILL, bool WIDE>
__global__ void __launch_bounds__(32 * kPlWarps) k_plist(int nrows, const int* __restrict__ arp,
                                                         const int* __restrict__ acol, const int* __restrict__ brp,
                                                         const int* __restrict__ bcol, const int* __restrict__ crp,
                                                         const int* __restrict__ ccol, int* __restrict__ cnt,
                                                         const int* __restrict__ place,
                                                         const long long* __restrict__ sptr,
                                                         int2* __restrict__ pairs) {
  __shared__ int pre_all[kPlWarps][33];
  __shared__ int bst_all[kPlWarps][32];
  __shared__ int col_all[kPlWarps][kPlCols];
  int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int* pre = pre_all[w];
  int* bst = bst_all[w];
  int* scol = WIDE ? col_all[0] : col_all[w];
  int nw = WIDE ? gridDim.x : gridDim.x * kPlWarps;
  for (int row = WIDE ? blockIdx.x : blockIdx.x * kPlWarps + w; row < nrows; row += nw) {
    int c0 = crp[row], c1 = crp[row + 1];
    // eight dependent L2 loads per product otherwise
    const bool staged = c1 - c0 <= (WIDE ? kPlCols * kPlWarps : kPlCols);
    if (WIDE) __syncthreads();  // the row before this one is done with the columns
    if (staged)
      for (int t = WIDE ? threadIdx.x : lane; t < c1 - c0; t += WIDE ? 32 * kPlWarps : 32) scol[t] = ccol[c0 + t];
    if (WIDE) __syncthreads();
    int a1 = arp[row + 1];
    for (int e0 = arp[row] + (WIDE ? 32 * w : 0); e0 < a1; e0 += WIDE ? 32 * kPlWarps : 32) {
      int e = e0 + lane;
      bool has = e < a1;
      int j = has ? acol[e] : 0;
      int b0 = has ? brp[j] : 0;
      int len = has ? brp[j + 1] - b0 : 0;
      int inc = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
      }
      int total = __shfl_sync(0xffffffffu, inc, 31);
      pre[lane + 1] = inc;
      if (lane == 0) pre[0] = 0;
      bst[lane] = b0;
      __syncwarp();
      for (int t = lane; t < total; t += 32) {
        int lo = 0, hi = 32;  // owner q of product t: pre[q] <= t < pre[q+1]
        while (hi - lo > 1) {
          int mid = (lo + hi) >> 1;
          if (pre[mid] <= t) lo = mid; else hi = mid;
        }
        int f = bst[lo] + (t - pre[lo]);
        int q = staged ? c0 + find_col(scol, 0, c1 - c0, bcol[f]) : find_col(ccol, c0, c1, bcol[f]);
        int slot = atomicAdd(&cnt[q], 1);
        if (FILL) {
          const int at = place[q];
          pairs[sptr[at / kSellC] + (long long)slot * kSellC + at % kSellC] = make_int2(e0 + lo, f);
        }
      }
      __syncwarp();
    }
  }
}

// The lists' layout from the entries' counts: a window of kSellSigma entries per block,
// bucketed by decreasing count (ties in any order: an entry's sum does not depend on its
// place).  place[q] is q's position, perm its inverse, slots the slices' sizes.
// Buckets: one per count below 256, above it 32 per power of two, so that a slice's padding
// stays within a 32nd of its entries; counts from 2^16 on share the first bucket.
constexpr int kPlBuckets = 512;
__device__ __forceinline__ int pl_bucket(int l) {
  if (l < 256) return kPlBuckets - 1 - l;
  const int e = 31 - __clz(l);
  return kPlBuckets - 1 - min(256 + ((e - 8) << 5) + ((l >> (e - 5)) & 31), kPlBuckets - 1);
}
__global__ void __launch_bounds__(kSellSigma) k_pl_shape(int nnz, const int* __restrict__ cnt, int nslice,
                                                         int* __restrict__ perm, int* __restrict__ place,
                                                         int* __restrict__ slots) {
  __shared__ int first[kPlBuckets], wsum[kPlBuckets / 32], wide[kSellSigma / kSellC];
  const int t = threadIdx.x, w0 = blockIdx.x * kSellSigma, q = w0 + t;
  const int l = q < nnz ? cnt[q] : 0, b = pl_bucket(l);
  if (t < kPlBuckets) first[t] = 0;
  if (t < kSellSigma / kSellC) wide[t] = 0;
  __syncthreads();
  const int rank = q < nnz ? atomicAdd(&first[b], 1) : 0;
  __syncthreads();
  int v = 0, inc = 0;
  if (t < kPlBuckets) {
    inc = v = first[t];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, inc, o);
      if ((t & 31) >= o) inc += u;
    }
    if ((t & 31) == 31) wsum[t >> 5] = inc;
  }
  __syncthreads();
  if (t < kPlBuckets) {
    for (int u = 0; u < (t >> 5); ++u) inc += wsum[u];
    first[t] = inc - v;
  }
  __syncthreads();
  if (q < nnz) {
    const int r = first[b] + rank;
    perm[w0 + r] = q;
    place[q] = w0 + r;
    atomicMax(&wide[r / kSellC], l);
  } else if (q < nslice * kSellC) {
    perm[q] = -1;  // entries fill the window's front: the places past them are the ones past nnz
  }
  __syncthreads();
  if (t < kSellSigma / kSellC && w0 / kSellC + t < nslice) slots[w0 / kSellC + t] = kSellC * wide[t];
}

// Insertion sort of each entry's pairs by A entry, a thread per entry in slot order.
__global__ void k_pl_sort(int nslice, const long long* __restrict__ sptr, int2* __restrict__ pairs) {
  const int lane = threadIdx.x & 31;
  for (int s = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < nslice; s += (gridDim.x * blockDim.x) >> 5) {
    int2* p = pairs + sptr[s] + lane;
    const int w = (int)((sptr[s + 1] - sptr[s]) / kSellC);
    for (int t = 1; t < w; ++t) {
      const int2 k = p[(long long)t * kSellC];
      if (k.x < 0) break;  // past the entry's end
      int v = t - 1;
      for (; v >= 0 && p[(long long)v * kSellC].x > k.x; --v) p[(long long)(v + 1) * kSellC] = p[(long long)v * kSellC];
      p[(long long)(v + 1) * kSellC] = k;
    }
  }
}

// The same for the entries of wide rows, which a block's warps file out of order: a warp
// per entry, up to kPlSort pairs ranked in shared memory (an A entry contributes one product
// to an entry of C, so the keys are distinct).  A longer entry is written anew, in order:
// the row's A entries 32 at a time, each looking for the entry's column in its B row.
// (64^3, setup with matching aggregates of 8 / of 1024 cells, those entries sorted by one
// lane: 110 / 48 ms, 67 and 22 of them here; 49 / 25 ms so.)
constexpr int kPlSort = 512;
__global__ void __launch_bounds__(32 * kPlWarps) k_pl_rank(int nrows, const int* __restrict__ arp,
                                                           const int* __restrict__ acol, const int* __restrict__ brp,
                                                           const int* __restrict__ bcol, const int* __restrict__ crp,
                                                           const int* __restrict__ ccol, int nnz,
                                                           const int* __restrict__ cnt, const int* __restrict__ place,
                                                           const long long* __restrict__ sptr,
                                                           int2* __restrict__ pairs) {
  __shared__ int2 a_all[kPlWarps][kPlSort];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int2* a = a_all[w];
  for (int q = blockIdx.x * kPlWarps + w; q < nnz; q += gridDim.x * kPlWarps) {
    const int len = cnt[q], at = place[q];
    if (len < 2) continue;
    int2* p = pairs + sptr[at / kSellC] + at % kSellC;
    if (len > kPlSort) {
      int row = 0, end = nrows;  // crp[row] <= q < crp[row + 1]
      while (end - row > 1) {
        const int mid = (row + end) >> 1;
        if (crp[mid] <= q) row = mid; else end = mid;
      }
      const int c = ccol[q], a1 = arp[row + 1];
      int t = 0;
      for (int e0 = arp[row]; e0 < a1; e0 += 32) {
        const int e = e0 + lane;
        int f = -1;
        if (e < a1) {
          const int b1 = brp[acol[e] + 1];
          f = find_col(bcol, brp[acol[e]], b1, c);
          if (f == b1 || bcol[f] != c) f = -1;
        }
        const unsigned m = __ballot_sync(0xffffffffu, f >= 0);
        if (f >= 0) p[(long long)(t + __popc(m & ((1u << lane) - 1))) * kSellC] = make_int2(e, f);
        t += __popc(m);
      }
      continue;
    }
    for (int t = lane; t < len; t += 32) a[t] = p[(long long)t * kSellC];
    __syncwarp();
    for (int t = lane; t < len; t += 32) {
      const int2 k = a[t];
      int r = 0;
      for (int v = 0; v < len; ++v) r += a[v].x < k.x;
      p[(long long)r * kSellC] = k;
    }
    __syncwarp();
  }
}

__global__ void k_sum_rows_ll(int n, const int* __restrict__ u, unsigned long long* __restrict__ out) {
  unsigned long long s = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) s += (unsigned)u[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(out, s);
}

// acc + the products of U columns of a slice from p on, all loads in flight together; of
// the first `left` of them if PRED (warp-uniform).  The multiply-add is explicit: a sum may
// not depend on which of these forms its pairs fall into (the slice's width decides).
template <class T, int U, bool PRED>
__device__ __forceinline__ T pl_sum(const int2* __restrict__ p, int left, const T* __restrict__ aval,
                                    const T* __restrict__ bval, T acc) {
  int2 k[U];
  T a[U], b[U];
#pragma unroll
  for (int u = 0; u < U; ++u) k[u] = !PRED || u < left ? __ldcs(&p[u * kSellC]) : make_int2(-1, 0);
#pragma unroll
  for (int u = 0; u < U; ++u) {
    a[u] = k[u].x >= 0 ? aval[k[u].x] : T(0);
    b[u] = k[u].x >= 0 ? bval[k[u].y] : T(0);
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (k[u].x >= 0) acc = fma(a[u], b[u], acc);
  return acc;
}

// c[q] = sum of a[x] * b[y] over q's pairs: no search, no atomics, the same sum every
// refresh.  A warp per slice, a thread per entry, four pairs in flight, summed in their order.
// Bound: FP64 one FMA per pair, FP32 HBM (8 bytes per pair).  128^3 FP64, 176M pairs over
// three levels: 1270 us with the pairs entry by entry (a thread's own run, 32 sectors per
// warp and load, and as many steps as the longest of 32 neighbours), 880 us so.
// SPLIT: a block per slice, for products whose slices are few and long, where a warp's chain
// of loads would be the time: its warps take the columns eight at a time in turn (an entry's
// split is its own, whatever slice it shares) and their sums are added in order.  All products
// of a refresh, FP64, without and so: 48^3 437 and 135 us, 96^3 918 and 512, 128^3 1289 and
// 1150; matching aggregates of 1024 cells on 64^3 657 and 227.
template <class T, bool SPLIT>
__global__ void __launch_bounds__(32 * kPlWarps) k_galerkin_lists(int nslice, const int* __restrict__ perm,
                                                                  const long long* __restrict__ sptr,
                                                                  const int2* __restrict__ pairs,
                                                                  const T* __restrict__ aval,
                                                                  const T* __restrict__ bval, T* __restrict__ cval) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (SPLIT) {
    __shared__ T part[kPlWarps][kSellC];
    const int s = blockIdx.x, q = perm[s * kSellC + lane];
    const int2* p = pairs + sptr[s] + lane;
    const int width = (int)((sptr[s + 1] - sptr[s]) / kSellC);
    T acc = T(0);
    for (int c = 8 * w; c < width; c += 8 * kPlWarps)
      acc = pl_sum<T, 8, true>(p + (long long)c * kSellC, width - c, aval, bval, acc);
    part[w][lane] = acc;
    __syncthreads();
    if (w > 0) return;
    for (int v = 1; v < kPlWarps; ++v) acc += part[v][lane];
    if (q >= 0) cval[q] = acc;
    return;
  }
  for (int s = blockIdx.x * kPlWarps + w; s < nslice; s += gridDim.x * kPlWarps) {
    // loaded ahead of the pairs: after them, entries of 3 products took 233 us for 190 (128^3)
    const int q = perm[s * kSellC + lane];
    const int2* p = pairs + sptr[s] + lane;
    const int2* end = pairs + sptr[s + 1];
    T acc = T(0);
    for (; p + 3 * kSellC < end; p += 4 * kSellC) acc = pl_sum<T, 4, false>(p, 4, aval, bval, acc);
    for (; p < end; p += kSellC) acc = pl_sum<T, 1, false>(p, 1, aval, bval, acc);
    if (q >= 0) cval[q] = acc;
  }
}

// ---------------------------------------------------------------- coarsest level: dense inverse

// Entries of a CSR matrix into a zeroed dense one, a warp per row.
template <class T>
__global__ void k_csr_to_dense(int n, const int* __restrict__ rp, const int* __restrict__ col,
                               const T* __restrict__ val, double* __restrict__ dense) {
  const int lane = threadIdx.x & 31;
  for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += (gridDim.x * blockDim.x) >> 5)
    for (int e = rp[i] + lane; e < rp[i + 1]; e += 32) dense[(long long)i * n + col[e]] = (double)val[e];
}

// Blocked Gauss-Jordan inversion in place (no pivoting: the matrix is SPD).
// For a panel P of kGjB consecutive pivots and the other indices O, one block
// step turns [[A_PP, A_PO], [A_OP, A_OO]] into
//   [[A_PP^-1, A_PP^-1 A_PO], [-A_OP A_PP^-1, A_OO - A_OP A_PP^-1 A_PO]];
// after every panel the matrix holds A^-1.  The matrix being symmetric, every step leaves
// a_ij = a_ji where both indices or neither has been a pivot and a_ij = -a_ji otherwise, so
// only the tiles on and above the diagonal are computed (n^3 / 2 multiply-adds instead of
// n^3) and mirrored; the upper triangle is what is inverted.  Two launches per panel:
// k_gj_rows forms the new panel rows (and their mirror), k_gj_update applies the rank-kGjB
// update, and its block on the next diagonal tile inverts that tile while the others are
// still at work.  Work buffer (2 kGjB n + kGjB^2 doubles): R[p][j] (new panel rows),
// C[p][i] (old panel columns), Pinv (kGjB x kGjB).
// Bound: FP64 multiply-adds for large n, the chain of pivots for small n.  n = 362: 713 us
// with full tiles, three launches per panel and a 42 us panel inversion.
constexpr int kGjB = 32;
constexpr int kGjInvWarps = 8;

// Inverse of the bs x bs block m by Gauss-Jordan in registers, by the first 8 warps of a
// block: warp w holds rows w, w + 8, w + 16, w + 24, a lane per column.  Per pivot the
// owner scales its row, one barrier publishes it (double buffer), and every other row takes
// one multiply-add; a column's factor comes from the pivot's lane by a shuffle.
__device__ __forceinline__ void gj_invert(double (*m)[kGjB + 1], int bs, double (*rk)[kGjB]) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double v[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int r = w + 8 * t;
    v[t] = r < bs && lane < bs ? m[r][lane] : (r == lane ? 1.0 : 0.0);
  }
#pragma unroll
  for (int t0 = 0; t0 < 4; ++t0) {
    for (int kk = 0; kk < 8; ++kk) {
      const int k = 8 * t0 + kk;
      if (k >= bs) break;
      double* row = rk[k & 1];
      if (w == kk) {
        const double inv = safe_rcp(__shfl_sync(0xffffffffu, v[t0], k));
        v[t0] = lane == k ? inv : v[t0] * inv;
        row[lane] = v[t0];
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      const double q = row[lane];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const double f = __shfl_sync(0xffffffffu, v[t], k);
        if (w + 8 * t != k) v[t] = fma(-f, q, lane == k ? 0.0 : v[t]);
      }
    }
  }
  asm volatile("bar.sync 1, 256;" ::: "memory");
#pragma unroll
  for (int t = 0; t < 4; ++t) m[w + 8 * t][lane] = v[t];
  asm volatile("bar.sync 1, 256;" ::: "memory");
}

// Inverse of the panel block at K: into the matrix and Pinv (zeros outside a partial block).
__device__ __forceinline__ void gj_store_panel(double (*m)[kGjB + 1], int n, int K, int bs, double* __restrict__ a,
                                               double* __restrict__ pinv) {
  for (int t = threadIdx.x; t < kGjB * kGjB; t += 32 * kGjInvWarps) {
    const int r = t / kGjB, q = t % kGjB;
    const bool in = r < bs && q < bs;
    if (in) a[(long long)(K + r) * n + K + q] = m[r][q];
    pinv[t] = in ? m[r][q] : 0.0;
  }
}

__global__ void __launch_bounds__(32 * kGjInvWarps) k_gj_panel(int n, int bs, double* __restrict__ a,
                                                              double* __restrict__ pinv) {
  __shared__ double m[kGjB][kGjB + 1], rk[2][kGjB];
  for (int t = threadIdx.x; t < kGjB * kGjB; t += 32 * kGjInvWarps) {
    const int r = t / kGjB, q = t % kGjB;
    m[r][q] = r < bs && q < bs ? a[(long long)min(r, q) * n + max(r, q)] : 0.0;
  }
  __syncthreads();
  gj_invert(m, bs, rk);
  gj_store_panel(m, n, 0, bs, a, pinv);
}

// Columns j0 .. j0+7 per block, thread (p, jj): R[p][j] = (Pinv A_P,j)_p to panel row p and,
// mirrored, to column p; C[p][j] = a_j,K+p before the step (a_K+p,j, negated for an earlier
// pivot j).  Columns in P take zeros (the panel itself is done).
constexpr int kGjCols = 8;

__global__ void __launch_bounds__(kGjB* kGjCols) k_gj_rows(int n, int K, int bs, double* __restrict__ a,
                                                          const double* __restrict__ pinv, double* __restrict__ R,
                                                          double* __restrict__ C) {
  __shared__ double ps[kGjB][kGjB + 1];
  __shared__ double cs[kGjB][kGjCols];
  __shared__ double out[kGjB][kGjCols + 1];
  const int p = threadIdx.x, jj = threadIdx.y;
  for (int t = jj; t < kGjB; t += kGjCols) ps[t][p] = pinv[t * kGjB + p];
  const int t = jj * kGjB + p, lr = t / kGjCols, lj = blockIdx.x * kGjCols + t % kGjCols;  // coalesced in j
  cs[lr][t % kGjCols] = (lj < n && lr < bs) ? a[(long long)(K + lr) * n + lj] : 0.0;
  __syncthreads();
  const int j = blockIdx.x * kGjCols + jj;
  const bool inP = j >= K && j < K + bs;
  double v = 0.0;
#pragma unroll
  for (int q = 0; q < kGjB; ++q) v = fma(ps[p][q], cs[q][jj], v);
  out[p][jj] = v;
  if (j < n && p < bs && !inP) a[(long long)j * n + K + p] = j < K ? v : -v;
  __syncthreads();
  if (lj >= n) return;
  const bool lp = lj >= K && lj < K + bs;
  const double w = out[lr][t % kGjCols], old = cs[lr][t % kGjCols];
  R[(long long)lr * n + lj] = lp ? 0.0 : w;
  C[(long long)lr * n + lj] = lp ? 0.0 : (lj < K ? -old : old);
  if (lr < bs && !lp) a[(long long)(K + lr) * n + lj] = w;
}

// a_ij -= sum_p C[p][i] R[p][j] for one kGjB x kGjB tile on or above the diagonal per
// block, outside the panel's row and column, and its mirror image; the block on the next
// diagonal tile inverts it.
__global__ void __launch_bounds__(kGjB* kGjB) k_gj_update(int n, int K, int bs, int nt, double* __restrict__ a,
                                                         const double* __restrict__ R, const double* __restrict__ C,
                                                         double* __restrict__ pinv) {
  __shared__ double cs[kGjB][kGjB + 1];  // cs[p][ti], then the tile
  __shared__ double rs[kGjB][kGjB + 1];  // rs[p][tj]
  __shared__ double rk[2][kGjB];
  // tile (I, J), I <= J, from the block number, rows of tiles in order; block 0 takes the
  // next diagonal tile, so that its inversion starts first
  const int kt = K / kGjB, next = kt + 1;
  int b = blockIdx.x, I = 0, J;
  if (next < nt) {  // number of (next, next) in the order
    const int nn = next * nt - next * (next - 1) / 2;
    if (b == 0) b = nn;
    else if (b <= nn) --b;
  }
  while (b >= nt - I) b -= nt - I++;
  J = I + b;
  if (I == kt || J == kt) return;
  const int tj = threadIdx.x & 31, ti = threadIdx.x >> 5;
  const int i0 = I * kGjB, j0 = J * kGjB;
  {
    const int i = i0 + tj, j = j0 + tj;
    cs[ti][tj] = (ti < bs && i < n) ? C[(long long)ti * n + i] : 0.0;
    rs[ti][tj] = (ti < bs && j < n) ? R[(long long)ti * n + j] : 0.0;
  }
  __syncthreads();
  const int i = i0 + ti, j = j0 + tj;
  const bool in = i < n && j < n;
  double acc = in ? a[(long long)i * n + j] : 0.0;
#pragma unroll 8
  for (int p = 0; p < kGjB; ++p) acc = fma(-cs[p][ti], rs[p][tj], acc);
  if (in) a[(long long)i * n + j] = acc;
  __syncthreads();
  cs[ti][tj] = acc;
  __syncthreads();
  if (I < J) {
    // pivots so far: tiles up to kt; the sign of the mirror image where only one has been
    const double s = (I <= kt) == (J <= kt) ? 1.0 : -1.0;
    const int mi = j0 + ti, mj = i0 + tj;
    if (mi < n && mj < n) a[(long long)mi * n + mj] = s * cs[tj][ti];
  } else if (I == next) {
    if (tj < ti) cs[ti][tj] = cs[tj][ti];
    __syncthreads();
    if (threadIdx.x < 32 * kGjInvWarps) {
      const int nbs = min(kGjB, n - i0);
      gj_invert(cs, nbs, rk);
      gj_store_panel(cs, n, i0, nbs, a, pinv);
    }
  }
}

// ---------------------------------------------------------------- matching aggregation
// Coupled aggregation by compatible weighted matching (the paper's SMATCH
// coarsening, Sec. 5.2).  Edge {i, j} of a negative coupling has the weight
// w_ij = 1 - (a_ij + a_ji) / (a_ii + a_jj) (smooth vector of ones), rounded to
// FP32 so that rounding-order differences of the FP64 matrices do not reorder
// equal weights; edges are ordered by weight, then by (min, max) index pair.
// The matching is locally dominant: synchronous rounds in which every unmatched
// node proposes to its best unmatched neighbour and mutual proposals match.

__device__ __forceinline__ bool match_better(float w1, int lo1, int hi1, float w2, int lo2, int hi2) {
  if (w1 != w2) return w1 > w2;
  if (lo1 != lo2) return lo1 < lo2;
  return hi1 < hi2;
}

__global__ void k_match_weights(int n, const int* __restrict__ rp, const int* __restrict__ col,
                                const double* __restrict__ val, const double* __restrict__ d,
                                float* __restrict__ w) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    for (int e = rp[i]; e < rp[i + 1]; ++e) {
      int j = col[e];
      float wv = -CUDART_INF_F;
      if (j != i) {
        int q = find_col(col, rp[j], rp[j + 1], i);  // a_ji (the pattern is symmetric)
        if (q < rp[j + 1] && col[q] == i) {
          double sum = val[e] + val[q];
          if (sum < 0.0) wv = (float)(1.0 - sum / (d[i] + d[j]));
        }
      }
      w[e] = wv;
    }
  }
}

// Proposals of one round; *any = 1 if some node proposed.
__global__ void k_match_propose(int n, const int* __restrict__ rp, const int* __restrict__ col,
                                const float* __restrict__ w, const int* __restrict__ mate, int* __restrict__ cand,
                                int* __restrict__ any) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int best = -1;
    float bw = -CUDART_INF_F;
    int blo = 0, bhi = 0;
    if (mate[i] < 0) {
      for (int e = rp[i]; e < rp[i + 1]; ++e) {
        int j = col[e];
        float we = w[e];
        if (we == -CUDART_INF_F || mate[j] >= 0) continue;
        int lo = min(i, j), hi = max(i, j);
        if (best < 0 || match_better(we, lo, hi, bw, blo, bhi)) {
          best = j;
          bw = we;
          blo = lo;
          bhi = hi;
        }
      }
    }
    cand[i] = best;
    if (best >= 0) *any = 1;
  }
}

__global__ void k_match_commit(int n, const int* __restrict__ cand, int* __restrict__ mate) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int j = cand[i];
    if (j >= 0 && cand[j] == i) mate[i] = j;
  }
}

// 1 for the smallest member of each pair and for every unmatched node.
__global__ void k_pair_first(int n, const int* __restrict__ mate, int* __restrict__ first) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    first[i] = mate[i] < 0 || i < mate[i];
}

__global__ void k_pair_ids(int n, const int* __restrict__ mate, const int* __restrict__ pos, int* __restrict__ ids) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int m = mate[i];
    ids[i] = pos[m < 0 ? i : min(i, m)];
  }
}

// agg[i] = ids[agg[i]] (composition of the pairing passes).
__global__ void k_compose(int n, const int* __restrict__ ids, int* __restrict__ agg) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) agg[i] = ids[agg[i]];
}

__global__ void k_iota(int n, int* __restrict__ a) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) a[i] = i;
}

// Single-pass SpGEMM: row r's cnt[r] compressed entries move from the temporary at
// its product offset uoff[r] to crp[r]; one warp per row.
__global__ void k_compact_rows(int n, const long long* __restrict__ uoff, const int* __restrict__ cnt,
                               const int* __restrict__ crp, const int* __restrict__ tcol,
                               const double* __restrict__ tval, int* __restrict__ ccol, double* __restrict__ cval) {
  const int lane = threadIdx.x & 31;
  for (long long row = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; row < n;
       row += ((long long)gridDim.x * blockDim.x) >> 5) {
    const long long src = uoff[row];
    const int dst = crp[row], m = cnt[row];
    for (int t = lane; t < m; t += 32) {
      ccol[dst + t] = tcol[src + t];
      cval[dst + t] = tval[src + t];
    }
  }
}

// ---------------------------------------------------------------- host side

// One int from the device, on the context's stream only (a plain cudaMemcpy would
// run on the legacy default stream and wait for every blocking stream, e.g. the
// other request-server slots).
static int read_dev_int(rich_ctx* c, const int* src, int* out) {
  RICH_CUDA(cudaMemcpyAsync(c->hflag + 8, src, sizeof(int), cudaMemcpyDeviceToHost, c->st));
  RICH_CUDA(cudaStreamSynchronize(c->st));
  *out = c->hflag[8];
  return RICH_OK;
}

static int spgemm_upper(rich_ctx* c, const Csr<double>& A, const Csr<double>& B, int* u, int* umax) {
  int n = A.nrows;
  k_spgemm_upper<<<grid_for(n), kBlock, 0, c->st>>>(n, A.rowptr, A.col, B.rowptr, u);
  RICH_LAUNCH_CHECK();
  if (umax) {
    RICH_CUDA(cudaMemsetAsync(c->iflag, 0, sizeof(int), c->st));
    k_max_int<<<grid_for(n), kBlock, 0, c->st>>>(n, u, c->iflag);
    RICH_LAUNCH_CHECK();
    RICH_CUDA(cudaMemcpyAsync(c->hflag, c->iflag, sizeof(int), cudaMemcpyDeviceToHost, c->st));
    RICH_CUDA(cudaStreamSynchronize(c->st));
    *umax = c->hflag[0];
  }
  return RICH_OK;
}

// C = A B: structural pattern (sorted columns) and values.  *u_keep, if given,
// receives the per-row product counts (kept for the numeric refresh); *hashed, if
// given, whether rows with more than kEscCap products went through the hash kernel,
// whose FP64 sums follow the order of shared-memory atomics.
static int spgemm_symbolic(rich_ctx* c, const Csr<double>& A, const Csr<double>& B, Csr<double>& C,
                           int** u_keep = nullptr, bool* hashed = nullptr) {
  int n = A.nrows;
  C.nrows = n;
  C.ncols = B.ncols;
  int* u = nullptr;
  int* cnt = nullptr;
  RICH_CHECK(dalloc(&u, n));
  RICH_CHECK(dalloc(&cnt, n));
  RICH_CHECK(dalloc(&C.rowptr, (long long)n + 1));
  int umax = 0;
  RICH_CHECK(spgemm_upper(c, A, B, u, &umax));
  if (umax >= (1 << 30)) return RICH_ELIMIT;
  // shared memory per warp sized by the largest row of this product
  int cap = 32;
  while (cap < umax && cap < kEscCap) cap <<= 1;
  const int esc_warps = cap <= 128 ? 8 : (cap <= 512 ? 4 : 2);
  size_t smem = (size_t)esc_warps * cap * (sizeof(uint64_t) + sizeof(double));
  int nblk = (n + esc_warps - 1) / esc_warps;
  if (nblk > 65535 * 4) nblk = 65535 * 4;
  bool big = umax > kEscCap;
  if (hashed) *hashed = big;
  size_t hsmem = (size_t)kHashSlots * (sizeof(int) + sizeof(double) + sizeof(uint64_t));
  if (big) RICH_CUDA(cudaFuncSetAttribute(k_spgemm_hash, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hsmem));
  int* ovf = c->iflag + 1;
  RICH_CUDA(cudaMemsetAsync(ovf, 0, sizeof(int), c->st));
  // One pass when a temporary of every product's slot fits in a quarter of the free
  // memory: each row is expanded, sorted and compressed once, at its product offset,
  // then compacted.  Otherwise two passes (count, then write at the final offsets).
  long long* uoff = nullptr;
  RICH_CHECK(dalloc(&uoff, (long long)n + 1));
  RICH_CHECK(scan_exclusive_int_ll(c, u, uoff, n));
  long long nprod = 0;
  RICH_CUDA(cudaMemcpyAsync(&nprod, uoff + n, sizeof(long long), cudaMemcpyDeviceToHost, c->st));
  RICH_CUDA(cudaStreamSynchronize(c->st));
  size_t mfree = 0, mtotal = 0;
  RICH_CUDA(cudaMemGetInfo(&mfree, &mtotal));
  mfree += pool_slack();
  const bool one_pass = (double)nprod * (sizeof(int) + sizeof(double)) <= 0.25 * (double)mfree;
  int* tcol = nullptr;
  double* tval = nullptr;
  if (one_pass) {
    RICH_CHECK(dalloc(&tcol, nprod));
    RICH_CHECK(dalloc(&tval, nprod));
  }
  for (int pass = 0; pass < 2; ++pass) {
    const int mode = one_pass ? 2 : pass;
    if (pass == 1) {
      // the row offsets are 32-bit: check the total in 64 bits before the scan
      unsigned long long* dsum = reinterpret_cast<unsigned long long*>(c->iflag + 4);  // slots 4-5
      RICH_CUDA(cudaMemsetAsync(dsum, 0, sizeof(unsigned long long), c->st));
      k_sum_rows_ll<<<red_grid(n), kBlock, 0, c->st>>>(n, cnt, dsum);
      RICH_LAUNCH_CHECK();
      unsigned long long total = 0;
      RICH_CUDA(cudaMemcpyAsync(&total, dsum, sizeof(total), cudaMemcpyDeviceToHost, c->st));
      RICH_CUDA(cudaStreamSynchronize(c->st));
      if (total > 2147483647ull) return RICH_ELIMIT;
      RICH_CHECK(scan_exclusive_int(c, cnt, C.rowptr, n));
      int nnz = 0;
      RICH_CHECK(read_dev_int(c, C.rowptr + n, &nnz));
      if (nnz < 0 || (unsigned long long)nnz != total) return RICH_ELIMIT;
      C.nnz = nnz;
      RICH_CHECK(dalloc(&C.col, nnz));
      RICH_CHECK(dalloc(&C.val, nnz));
      if (one_pass) {
        k_compact_rows<<<grid_for(32LL * n), kBlock, 0, c->st>>>(n, uoff, cnt, C.rowptr, tcol, tval, C.col, C.val);
        RICH_LAUNCH_CHECK();
        break;
      }
    }
    int* ocol = mode == 2 ? tcol : C.col;
    double* oval = mode == 2 ? tval : C.val;
    if (B.ncols < (1 << kSortCol)) {
      auto run = [&](auto kernel, int umin, int cp, int wpb) -> int {
        if (umin >= cap) return RICH_OK;
        cp = std::min(cap, cp);
        const int nblk2 = std::min((n + wpb - 1) / wpb, 64 * kNumSM);
        kernel<<<nblk2, 32 * wpb, (size_t)wpb * cp * (sizeof(double) + sizeof(unsigned)), c->st>>>(
            n, A.rowptr, A.col, A.val, B.rowptr, B.col, B.val, u, mode, C.rowptr, uoff, ocol, oval, cnt, umin, cp);
        RICH_LAUNCH_CHECK();
        return RICH_OK;
      };
      RICH_CHECK(run(k_spgemm_sort<2>, 0, 64, 8));
      RICH_CHECK(run(k_spgemm_sort<8>, 64, 256, 8));
      RICH_CHECK(run(k_spgemm_sort<32>, 256, 1024, cap <= 512 ? 4 : 2));
    } else {
      k_spgemm_esc<<<nblk, 32 * esc_warps, smem, c->st>>>(n, A.rowptr, A.col, A.val, B.rowptr, B.col, B.val, u, mode,
                                                         C.rowptr, uoff, ocol, oval, cnt, cap);
      RICH_LAUNCH_CHECK();
    }
    if (big) {
      int hb = n < 8 * kNumSM ? n : 8 * kNumSM;
      k_spgemm_hash<<<hb, kHashThreads, hsmem, c->st>>>(n, A.rowptr, A.col, A.val, B.rowptr, B.col, B.val, u, mode,
                                                        C.rowptr, uoff, ocol, oval, cnt, ovf);
      RICH_LAUNCH_CHECK();
      RICH_CUDA(cudaMemcpyAsync(c->hflag + 1, ovf, sizeof(int), cudaMemcpyDeviceToHost, c->st));
      RICH_CUDA(cudaStreamSynchronize(c->st));
      if (c->hflag[1]) return RICH_ELIMIT;  // a row has more distinct columns than the hash table holds
    }
  }
  dfree(tcol);
  dfree(tval);
  dfree(uoff);
  if (u_keep) *u_keep = u; else dfree(u);
  dfree(cnt);
  return RICH_OK;
}

static const char* kNumericName[2][16] = {
    {"galerkin_ap_l0", "galerkin_ap_l1", "galerkin_ap_l2", "galerkin_ap_l3", "galerkin_ap_l4", "galerkin_ap_l5",
     "galerkin_ap_l6", "galerkin_ap_l7", "galerkin_ap_l8", "galerkin_ap_l9", "galerkin_ap", "galerkin_ap",
     "galerkin_ap", "galerkin_ap", "galerkin_ap", "galerkin_ap"},
    {"galerkin_rap_l0", "galerkin_rap_l1", "galerkin_rap_l2", "galerkin_rap_l3", "galerkin_rap_l4",
     "galerkin_rap_l5", "galerkin_rap_l6", "galerkin_rap_l7", "galerkin_rap_l8", "galerkin_rap_l9", "galerkin_rap",
     "galerkin_rap", "galerkin_rap", "galerkin_rap", "galerkin_rap", "galerkin_rap"}};

static void plist_free(ProdList& pl) {
  dfree(pl.perm);
  dfree(pl.sptr);
  dfree(pl.pairs);
  pl.nslice = 0;
  pl.np = 0;
}

// Product lists of C = A B (u = products per row).  Leaves pl empty, and
// returns RICH_OK, when the lists would not fit in half the free device
// memory; the refresh then falls back to the searching kernels.
static int plist_build(rich_ctx* c, const Csr<double>& A, const Csr<double>& B, const Csr<double>& C, const int* u,
                       ProdList& pl) {
  plist_free(pl);
  unsigned long long* dsum = reinterpret_cast<unsigned long long*>(c->iflag + 4);  // slots 4-5, 16-byte aligned
  RICH_CUDA(cudaMemsetAsync(dsum, 0, sizeof(unsigned long long), c->st));
  k_sum_rows_ll<<<red_grid(A.nrows), kBlock, 0, c->st>>>(A.nrows, u, dsum);
  RICH_LAUNCH_CHECK();
  unsigned long long np = 0;
  RICH_CUDA(cudaMemcpyAsync(&np, dsum, sizeof(np), cudaMemcpyDeviceToHost, c->st));
  RICH_CUDA(cudaStreamSynchronize(c->st));
  size_t fr = 0, tot = 0;
  RICH_CUDA(cudaMemGetInfo(&fr, &tot));
  fr += pool_slack();  // blocks freed into the pool count as free here
  if (!plist_fits((double)np, (double)C.nnz, (double)fr)) return RICH_OK;
  const int nnz = (int)C.nnz;
  pl.nslice = (nnz + kSellC - 1) / kSellC;
  int *cnt = nullptr, *place = nullptr, *slots = nullptr;
  RICH_CHECK(dalloc(&cnt, nnz + 1LL));
  RICH_CHECK(dalloc(&place, nnz + 1LL));
  RICH_CHECK(dalloc(&slots, pl.nslice));
  RICH_CHECK(dalloc(&pl.perm, (long long)pl.nslice * kSellC));
  RICH_CHECK(dalloc(&pl.sptr, pl.nslice + 1LL));
  pl.np = (long long)np;
  const bool wide = (double)np > 512.0 * A.nrows;
  int nwb = wide ? A.nrows : (A.nrows + kPlWarps - 1) / kPlWarps;
  if (nwb > 64 * kNumSM) nwb = 64 * kNumSM;
  auto list = [&](auto kernel) {
    kernel<<<nwb, 32 * kPlWarps, 0, c->st>>>(A.nrows, A.rowptr, A.col, B.rowptr, B.col, C.rowptr, C.col, cnt, place,
                                             pl.sptr, pl.pairs);
  };
  RICH_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int) * ((size_t)nnz + 1), c->st));
  if (wide) list(k_plist<false, true>);
  else list(k_plist<false, false>);
  RICH_LAUNCH_CHECK();
  k_pl_shape<<<(nnz + kSellSigma - 1) / kSellSigma, kSellSigma, 0, c->st>>>(nnz, cnt, pl.nslice, pl.perm, place, slots);
  RICH_LAUNCH_CHECK();
  RICH_CHECK(scan_exclusive_int_ll(c, slots, pl.sptr, pl.nslice));
  long long total = 0;
  RICH_CUDA(cudaMemcpyAsync(&total, pl.sptr + pl.nslice, sizeof(total), cudaMemcpyDeviceToHost, c->st));
  RICH_CUDA(cudaStreamSynchronize(c->st));
  if (!plist_fits((double)total, (double)C.nnz, (double)fr)) {  // padded beyond the limit: the refresh searches
    plist_free(pl);
  } else if (dalloc(&pl.pairs, total) != RICH_OK) {  // or beyond what is left
    cudaGetLastError();
    plist_free(pl);
  } else {
    RICH_CUDA(cudaMemsetAsync(pl.pairs, 0xff, sizeof(int2) * (size_t)total, c->st));  // x = -1: no pair
    RICH_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int) * ((size_t)nnz + 1), c->st));
    if (wide) list(k_plist<true, true>);
    else list(k_plist<true, false>);
    RICH_LAUNCH_CHECK();
    // entries filed by one warp per row are almost in order already
    if (wide)
      k_pl_rank<<<std::min((nnz + kPlWarps - 1) / kPlWarps, 64 * kNumSM), 32 * kPlWarps, 0, c->st>>>(
          A.nrows, A.rowptr, A.col, B.rowptr, B.col, C.rowptr, C.col, nnz, cnt, place, pl.sptr, pl.pairs);
    else
      k_pl_sort<<<grid_for(32LL * pl.nslice), kBlock, 0, c->st>>>(pl.nslice, pl.sptr, pl.pairs);
    RICH_LAUNCH_CHECK();
  }
  dfree(cnt);
  dfree(place);
  dfree(slots);
  return RICH_OK;
}

// C = A B on C's pattern with values of type T (aval/bval/cval); which = 0 for
// A P, 1 for R (A P); level for the profile name.  pl, if it holds lists, is used.
template <class T>
static int spgemm_numeric_t(rich_ctx* c, const Csr<double>& A, const T* aval, const Csr<double>& B, const T* bval,
                            const Csr<double>& C, T* cval, const int* u, int which, int level,
                            const ProdList* pl = nullptr) {
  if (pl && pl->built()) {
    ProfScope ps(kNumericName[which][level & 15], c->st,
                 4.0 * ((double)C.nnz + 1) + 8.0 * (double)pl->np +
                     (double)sizeof(T) * ((double)A.nnz + (double)B.nnz + (double)C.nnz),
                 2.0 * (double)pl->np);
    auto run = [&](auto kernel, int blocks) {
      kernel<<<blocks, 32 * kPlWarps, 0, c->st>>>(pl->nslice, pl->perm, pl->sptr, pl->pairs, aval, bval, cval);
    };
    // A warp per slice does not hide its loads' latency while there are few of them, the longer
    // the entries the more are few.  FP64, a warp and a block per slice: entries of 9 products in
    // 68 slices per SM 43 and 29 us, in 91 per SM 35 and 40; of 30 products in 77 per SM 174 and
    // 62, in 320 per SM 283 and 230, in 620 per SM 444 and 442 (FP32 328 and 342).  A pair or two
    // per warp (entries of 3 products) is not worth it.
    const double len = (double)pl->np / (double)C.nnz;
    if (pl->nslice < (len > 20.0 ? 320 : len > 8.0 ? 72 : 0) * kNumSM)
      run(k_galerkin_lists<T, true>, pl->nslice);
    else
      run(k_galerkin_lists<T, false>, grid_for(32LL * pl->nslice));
    RICH_LAUNCH_CHECK();
    return RICH_OK;
  }
  ProfScope ps(kNumericName[which][level & 15], c->st,
               (double)A.nrows * 4 + A.nnz * (4.0 + sizeof(T)) + (double)C.nrows * 4 + C.nnz * (4.0 + sizeof(T)));
  k_spgemm_numeric<T><<<grid_for(A.nrows, 128), 128, 0, c->st>>>(A.nrows, A.rowptr, A.col, aval, B.rowptr, B.col,
                                                                 bval, C.rowptr, C.col, cval, u);
  RICH_LAUNCH_CHECK();
  {
    int nwb = (A.nrows + kWarpRowsPerBlock - 1) / kWarpRowsPerBlock;
    if (nwb > 32 * kNumSM) nwb = 32 * kNumSM;
    k_spgemm_numeric_warp<T><<<nwb, 32 * kWarpRowsPerBlock, 0, c->st>>>(A.nrows, A.rowptr, A.col, aval, B.rowptr,
                                                                        B.col, bval, C.rowptr, C.col, cval, u);
    RICH_LAUNCH_CHECK();
  }
  int nb = A.nrows < 8 * kNumSM ? A.nrows : 8 * kNumSM;
  if (C.ncols <= kDenseCols) {
    const int dsm = (int)((kDenseCols + kNumAmax) * sizeof(double) + (kNumLmax + 2 * kNumAmax + 1) * sizeof(int));
    RICH_CUDA(cudaFuncSetAttribute(k_spgemm_numeric_block<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, dsm));
    k_spgemm_numeric_block<T, true><<<nb, kNumThreads, dsm, c->st>>>(A.nrows, A.rowptr, A.col, aval, B.rowptr, B.col,
                                                                    bval, C.rowptr, C.col, cval, u, C.ncols);
  } else {
    const int dsm = (int)((kNumLmax + kNumAmax) * sizeof(double) + (kNumLmax + 2 * kNumAmax + 1) * sizeof(int));
    RICH_CUDA(cudaFuncSetAttribute(k_spgemm_numeric_block<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, dsm));
    k_spgemm_numeric_block<T, false><<<nb, kNumThreads, dsm, c->st>>>(A.nrows, A.rowptr, A.col, aval, B.rowptr,
                                                                     B.col, bval, C.rowptr, C.col, cval, u, C.ncols);
  }
  RICH_LAUNCH_CHECK();
  return RICH_OK;
}

static int spgemm_numeric(rich_ctx* c, const Csr<double>& A, const Csr<double>& B, Csr<double>& C, const int* u,
                          int which = 0, int level = 0, const ProdList* pl = nullptr) {
  return spgemm_numeric_t<double>(c, A, A.val, B, B.val, C, C.val, u, which, level, pl);
}

static void csr_free(Csr<double>& m, bool pattern = true) {
  if (pattern) {
    dfree(m.rowptr);
    dfree(m.col);
  }
  dfree(m.val);
  m.nnz = 0;
}

static int identity_csr(rich_ctx* c, int m, Csr<double>& I) {
  I.nrows = I.ncols = m;
  I.nnz = m;
  RICH_CHECK(dalloc(&I.rowptr, (long long)m + 1));
  RICH_CHECK(dalloc(&I.col, m));
  I.val = nullptr;  // treated as all-ones by the ESC kernel
  k_seq<<<grid_for(m + 1), kBlock, 0, c->st>>>(m, I.rowptr);
  RICH_LAUNCH_CHECK();
  k_seq<<<grid_for(m), kBlock, 0, c->st>>>(m - 1, I.col);
  RICH_LAUNCH_CHECK();
  return RICH_OK;
}

// R = P^T with sorted columns (atomic placement, then a sort through R_unsorted * I)
static int transpose(rich_ctx* c, const Csr<double>& P, Csr<double>& R) {
  int n = P.nrows, m = P.ncols;
  Csr<double> T;
  T.nrows = m;
  T.ncols = n;
  T.nnz = P.nnz;
  int* cnt = nullptr;
  int* fillc = nullptr;
  RICH_CHECK(dalloc(&cnt, m));
  RICH_CHECK(dalloc(&fillc, m));
  RICH_CHECK(dalloc(&T.rowptr, (long long)m + 1));
  RICH_CHECK(dalloc(&T.col, P.nnz));
  RICH_CHECK(dalloc(&T.val, P.nnz));
  RICH_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int) * m, c->st));
  RICH_CUDA(cudaMemsetAsync(fillc, 0, sizeof(int) * m, c->st));
  k_tr_count<<<grid_for(n), kBlock, 0, c->st>>>(n, P.rowptr, P.col, cnt);
  RICH_LAUNCH_CHECK();
  RICH_CHECK(scan_exclusive_int(c, cnt, T.rowptr, m));
  k_tr_fill<<<grid_for(n), kBlock, 0, c->st>>>(n, P.rowptr, P.col, P.val, T.rowptr, fillc, T.col, T.val);
  RICH_LAUNCH_CHECK();
  Csr<double> I;
  RICH_CHECK(identity_csr(c, n, I));
  RICH_CHECK(spgemm_symbolic(c, T, I, R));
  csr_free(T);
  csr_free(I);
  dfree(cnt);
  dfree(fillc);
  return RICH_OK;
}

static int coarse_inverse_launches(rich_ctx* c);

// The coarsest inverse is n_c pivot launches; they are recorded once per hierarchy
// into a CUDA graph (fixed buffers) and replayed on every refresh.
static int coarse_inverse(rich_ctx* c) {
  Hierarchy& H = c->H;
  if (!H.dense) return RICH_OK;
  if (H.gj_exec) {
    ProfScope ps("coarse_inverse", c->st, 8.0 * (double)H.cn * H.cn * 2.0);
    RICH_CUDA(cudaGraphLaunch(H.gj_exec, c->st));
    count_launches(H.gj_nodes);
    return RICH_OK;
  }
  return coarse_inverse_launches(c);
}

static int capture_coarse_graph(rich_ctx* c) {
  Hierarchy& H = c->H;
  if (!H.dense || H.gj_exec) return RICH_OK;
  cudaStream_t cs;
  RICH_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
  cudaStream_t saved = c->st;
  RICH_CUDA(cudaStreamSynchronize(saved));
  c->st = cs;
  cudaGraph_t graph = nullptr;
  long long before = 0;
  rich_kernel_launches(&before);
  int rc = RICH_OK;
  cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    rc = coarse_inverse_launches(c);
    e = cudaStreamEndCapture(cs, &graph);
  }
  c->st = saved;
  long long after = 0;
  rich_kernel_launches(&after);
  count_launches(before - after);  // recorded, not launched
  if (e == cudaSuccess && rc == RICH_OK) {
    e = cudaGraphInstantiate(&H.gj_exec, graph, 0);
    if (e == cudaSuccess) H.gj_nodes = after - before;
    else H.gj_exec = nullptr;
  }
  if (graph) cudaGraphDestroy(graph);
  cudaStreamDestroy(cs);
  if (e != cudaSuccess) {
    cudaGetLastError();  // fall back to direct launches
    H.gj_exec = nullptr;
  }
  return rc;
}

static int coarse_inverse_launches(rich_ctx* c) {
  Hierarchy& H = c->H;
  Level& L = H.lv[H.nlev - 1];
  int n = L.n;
  long long nn = (long long)n * n;
  RICH_CUDA(cudaMemsetAsync(H.cdense, 0, sizeof(double) * (size_t)nn, c->st));
  // in MIXED precision the refreshed coarse values are the FP32 ones
  if (c->prec == RICH_PREC_MIXED && H.nlev > 1)
    k_csr_to_dense<float><<<grid_for(32LL * n), kBlock, 0, c->st>>>(n, L.A.rowptr, L.A.col, L.A32, H.cdense);
  else
    k_csr_to_dense<double><<<grid_for(32LL * n), kBlock, 0, c->st>>>(n, L.A.rowptr, L.A.col, L.A.val, H.cdense);
  RICH_LAUNCH_CHECK();
  double* R = H.cwork;
  double* C = R + (long long)kGjB * n;
  double* pinv = C + (long long)kGjB * n;
  const int nt = (n + kGjB - 1) / kGjB;
  k_gj_panel<<<1, 32 * kGjInvWarps, 0, c->st>>>(n, std::min(kGjB, n), H.cdense, pinv);
  RICH_LAUNCH_CHECK();
  for (int K = 0; K < n && nt > 1; K += kGjB) {
    const int bs = n - K < kGjB ? n - K : kGjB;
    k_gj_rows<<<(n + kGjCols - 1) / kGjCols, dim3(kGjB, kGjCols), 0, c->st>>>(n, K, bs, H.cdense, pinv, R, C);
    RICH_LAUNCH_CHECK();
    k_gj_update<<<nt * (nt + 1) / 2, kGjB * kGjB, 0, c->st>>>(n, K, bs, nt, H.cdense, R, C, pinv);
    RICH_LAUNCH_CHECK();
  }
  if (H.cinv32) {
    k_cast<<<grid_for(nn), kBlock, 0, c->st>>>(nn, H.cdense, H.cinv32);
    RICH_LAUNCH_CHECK();
  }
  return RICH_OK;
}

// Finest-level stencil arrays from the 7n diffusion stencil; dinv = 1 / (l1 row norm)
// = 1 / (diag + sum of the six face weights).
__global__ void k_stencil4(long long n, const double* __restrict__ A7, Stencil4<double> s64, Stencil4<float> s32) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    double a = A7[i], x = -A7[2 * n + i], y = -A7[4 * n + i], z = -A7[6 * n + i];
    double l1 = a + ((-A7[1 * n + i] + x) + (-A7[3 * n + i] + y) + (-A7[5 * n + i] + z));
    double r = 1.0 / l1;
    if (s64.diag) { s64.diag[i] = a; s64.wx[i] = x; s64.wy[i] = y; s64.wz[i] = z; s64.dinv[i] = r; }
    if (s32.diag) {
      s32.diag[i] = (float)a; s32.wx[i] = (float)x; s32.wy[i] = (float)y; s32.wz[i] = (float)z;
      s32.dinv[i] = (float)r;
    }
  }
}

// s = l1^-1/2 and q = l1^1/2 of every row, kept in FP64 for k_scaled.
__global__ void k_scale_rows(long long n, const double* __restrict__ A7, double* __restrict__ s, double* __restrict__ q,
                             float* __restrict__ s32, float* __restrict__ q32) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    double l1 = A7[i];
#pragma unroll
    for (int f = 1; f < 7; ++f) l1 -= A7[f * n + i];
    const double r = rsqrt(l1);
    s[i] = r;
    const double p = l1 * r;
    if (q) q[i] = p;
    if (s32) {
      s32[i] = (float)r;
      q32[i] = (float)p;
    }
  }
}

template <class T>
__global__ void k_scaled(GridP gr, const double* __restrict__ A7, const double* __restrict__ s, ScaledSt<T> A) {
  const int i = blockIdx.y * kLineThreads + threadIdx.x;
  if (i >= gr.nx) return;
  const long long n = gr.n, c = (long long)blockIdx.x * gr.nx + i;
  const int j = blockIdx.x % gr.ny, k = blockIdx.x / gr.ny, sxy = gr.nx * gr.ny;
  const double sc = s[c];
  const double d = -A7[c] * sc * sc;
  A.g[c] = (T)(1.0 + d);
  A.gd[c] = (T)d;
  A.wx[c] = i < gr.nx - 1 ? (T)(-A7[2 * n + c] * sc * s[c + 1]) : T(0);
  A.wy[c] = j < gr.ny - 1 ? (T)(-A7[4 * n + c] * sc * s[c + gr.nx]) : T(0);
  A.wz[c] = k < gr.nz - 1 ? (T)(-A7[6 * n + c] * sc * s[c + sxy]) : T(0);
}

template <class T>
static int scaled_alloc(ScaledSt<T>& A, long long n) {
  if (A.g) return RICH_OK;
  for (T** p : {&A.g, &A.gd, &A.wx, &A.wy, &A.wz, &A.s, &A.q}) RICH_CHECK(dalloc(p, n));
  return RICH_OK;
}
template <class T>
static void scaled_free(ScaledSt<T>& A) {
  for (T** p : {&A.g, &A.gd, &A.wx, &A.wy, &A.wz, &A.s, &A.q}) dfree(*p);
}

static int fine_scaled(rich_ctx* c) {
  Hierarchy& H = c->H;
  const long long n = c->g.n;
  if (c->prec == RICH_PREC_MIXED) {
    RICH_CHECK(scaled_alloc(H.sc32, n));
    if (!H.sc64.s) RICH_CHECK(dalloc(&H.sc64.s, n));  // FP64 factors for the weights' products
    k_scale_rows<<<grid_for(n), kBlock, 0, c->st>>>(n, c->A7, H.sc64.s, nullptr, H.sc32.s, H.sc32.q);
    RICH_LAUNCH_CHECK();
    k_scaled<float><<<line_grid(c->g), kLineThreads, 0, c->st>>>(c->g, c->A7, H.sc64.s, H.sc32);
  } else {
    RICH_CHECK(scaled_alloc(H.sc64, n));
    k_scale_rows<<<grid_for(n), kBlock, 0, c->st>>>(n, c->A7, H.sc64.s, H.sc64.q, nullptr, nullptr);
    RICH_LAUNCH_CHECK();
    k_scaled<double><<<line_grid(c->g), kLineThreads, 0, c->st>>>(c->g, c->A7, H.sc64.s, H.sc64);
  }
  RICH_LAUNCH_CHECK();
  return RICH_OK;
}

// Finest-level stencil copy of the diffusion matrix for the V-cycle (FP64 or FP32).
static int fine_stencil(rich_ctx* c) {
  Hierarchy& H = c->H;
  if (H.scaled) return fine_scaled(c);
  long long n = c->g.n;
  bool mp = c->prec == RICH_PREC_MIXED;
  if (mp && !H.st32.diag) {
    RICH_CHECK(dalloc(&H.st32.diag, n));
    RICH_CHECK(dalloc(&H.st32.wx, n));
    RICH_CHECK(dalloc(&H.st32.wy, n));
    RICH_CHECK(dalloc(&H.st32.wz, n));
    RICH_CHECK(dalloc(&H.st32.dinv, n));
  }
  if (!mp && !H.st64.diag) {
    RICH_CHECK(dalloc(&H.st64.diag, n));
    RICH_CHECK(dalloc(&H.st64.wx, n));
    RICH_CHECK(dalloc(&H.st64.wy, n));
    RICH_CHECK(dalloc(&H.st64.wz, n));
    RICH_CHECK(dalloc(&H.st64.dinv, n));
  }
  k_stencil4<<<grid_for(n), kBlock, 0, c->st>>>(n, c->A7, H.st64, H.st32);
  RICH_LAUNCH_CHECK();
  return RICH_OK;
}

// l1: the level's sweeps read 1/l1 (a scaled finest level's read ScaledSt instead); cast: the
// FP32 values, which MIXED's products and sweeps read.
static int level_diag_data(rich_ctx* c, Level& L, bool l1 = true, bool cast = true) {
  bool mp = c->prec == RICH_PREC_MIXED;
  if (l1) {
    k_l1dinv<<<grid_for(L.n), kBlock, 0, c->st>>>(L.n, L.A.rowptr, L.A.val, L.dinv, mp ? L.dinv32 : nullptr);
    RICH_LAUNCH_CHECK();
  }
  if (mp && cast) {
    k_cast<<<grid_for(L.A.nnz), kBlock, 0, c->st>>>(L.A.nnz, L.A.val, L.A32);
    RICH_LAUNCH_CHECK();
  }
  return RICH_OK;
}

// Values of level L's SELL copy of A (if the V-cycle has laid one out) from the
// values the V-cycle uses (FP32 in MIXED).
static int sell_fill_a(rich_ctx* c, Level& L) {
  if (c->prec == RICH_PREC_MIXED) return sell_fill(c, L.A, L.A32, L.sA);
  return sell_fill(c, L.A, L.A.val, L.sA);
}

static int level_alloc_vectors(rich_ctx* c, Level& L) {
  size_t es = c->prec == RICH_PREC_MIXED ? sizeof(float) : sizeof(double);
  long long n = L.n > 0 ? L.n : 1;
  void** vecs[4] = {&L.x, &L.b, &L.r, &L.t};
  for (void** v : vecs) {
    char* m = nullptr;
    RICH_CHECK(dalloc(&m, (long long)es * n));
    *v = m;
  }
  RICH_CHECK(dalloc(&L.dinv, n));
  if (c->prec == RICH_PREC_MIXED) {
    RICH_CHECK(dalloc(&L.dinv32, n));
    RICH_CHECK(dalloc(&L.A32, L.A.nnz));
  }
  return RICH_OK;
}

void amg_free(rich_ctx* c) {
  Hierarchy& H = c->H;
  for (int l = 0; l < (int)H.lv.size(); ++l) {
    Level& L = H.lv[l];
    if (l > 0) csr_free(L.A);
    csr_free(L.P);
    csr_free(L.R);
    csr_free(L.AP);
    dfree(L.A32);
    dfree(L.dinv);
    dfree(L.dinv32);
    dfree(L.agg);
    dfree(L.P32);
    dfree(L.R32);
    dfree(L.AP32);
    plist_free(L.pl_ap);
    plist_free(L.pl_rap);
    sell_free(L.sA);
    sell_free(L.sP);
    sell_free(L.sR);
    L.pl_tried = false;
    dfree(L.u_ap);
    dfree(L.u_rap);
    void** vecs[4] = {&L.x, &L.b, &L.r, &L.t};
    for (void** v : vecs) {
      char* m = static_cast<char*>(*v);
      dfree(m);
      *v = nullptr;
    }
  }
  H.lv.clear();
  H.nlev = 0;
  dfree(H.st64.diag); dfree(H.st64.wx); dfree(H.st64.wy); dfree(H.st64.wz); dfree(H.st64.dinv);
  dfree(H.st32.diag); dfree(H.st32.wx); dfree(H.st32.wy); dfree(H.st32.wz); dfree(H.st32.dinv);
  scaled_free(H.sc64);
  scaled_free(H.sc32);
  H.scaled = false;
  dfree(H.cdense);
  dfree(H.cinv32);
  dfree(H.cwork);
  if (H.gj_exec) cudaGraphExecDestroy(H.gj_exec);
  H.gj_exec = nullptr;
  H.gj_nodes = 0;
  if (H.vc_exec) cudaGraphExecDestroy(H.vc_exec);
  H.vc_exec = nullptr;
  H.vc_nodes = 0;
  H.vc_out = nullptr;
  H.vc_calls = 0;
  H.vc_off = false;
  for (int q = 0; q < 2; ++q) {
    if (H.fcg_exec[q]) cudaGraphExecDestroy(H.fcg_exec[q]);
    H.fcg_exec[q] = nullptr;
    H.fcg_nodes[q] = 0;
  }
  H.fcg_off = false;
  as_free(c);
  H.built = false;
}


// Coarsen level L into a new level; returns RICH_OK with *stop = true when coarsening stops.
// Aggregates of at most max_size nodes by log2(max_size) matching passes on A
// (the first pass) and on the successive pair graphs P_p^T A P_p.  agg (n ints)
// receives the aggregate of every node, *nc their number, *rounds the matching
// rounds summed over the passes.
static int matching_aggregate(rich_ctx* c, const Csr<double>& A, int max_size, int* agg, int* nc, int* rounds) {
  int n = A.nrows;
  int passes = 0;
  while ((2 << passes) <= max_size) ++passes;
  k_iota<<<grid_for(n), kBlock, 0, c->st>>>(n, agg);
  RICH_LAUNCH_CHECK();
  *nc = n;
  *rounds = 0;
  Csr<double> Ak = A;  // the first pass reads A itself
  bool own = false;
  for (int pass = 0; pass < passes; ++pass) {
    int m = Ak.nrows;
    double* d = nullptr;
    float* w = nullptr;
    int *mate = nullptr, *cand = nullptr, *first = nullptr, *pos = nullptr, *ids = nullptr;
    RICH_CHECK(dalloc(&d, m));
    RICH_CHECK(dalloc(&w, Ak.nnz));
    RICH_CHECK(dalloc(&mate, m));
    RICH_CHECK(dalloc(&cand, m));
    RICH_CHECK(dalloc(&first, m));
    RICH_CHECK(dalloc(&pos, (long long)m + 1));
    RICH_CHECK(dalloc(&ids, m));
    k_diag<<<grid_for(m), kBlock, 0, c->st>>>(m, Ak.rowptr, Ak.col, Ak.val, d);
    RICH_LAUNCH_CHECK();
    k_match_weights<<<grid_for(m), kBlock, 0, c->st>>>(m, Ak.rowptr, Ak.col, Ak.val, d, w);
    RICH_LAUNCH_CHECK();
    RICH_CUDA(cudaMemsetAsync(mate, 0xff, sizeof(int) * (size_t)m, c->st));  // -1: unmatched
    for (;;) {
      RICH_CUDA(cudaMemsetAsync(c->iflag, 0, sizeof(int), c->st));
      k_match_propose<<<grid_for(m), kBlock, 0, c->st>>>(m, Ak.rowptr, Ak.col, w, mate, cand, c->iflag);
      RICH_LAUNCH_CHECK();
      int any = 0;
      RICH_CHECK(read_dev_int(c, c->iflag, &any));
      if (!any) break;
      k_match_commit<<<grid_for(m), kBlock, 0, c->st>>>(m, cand, mate);
      RICH_LAUNCH_CHECK();
      ++*rounds;
      if (*rounds > 1000000) return RICH_ELIMIT;  // every round matches the globally best free edge
    }
    k_pair_first<<<grid_for(m), kBlock, 0, c->st>>>(m, mate, first);
    RICH_LAUNCH_CHECK();
    RICH_CHECK(scan_exclusive_int(c, first, pos, m));
    int mc = 0;
    RICH_CHECK(read_dev_int(c, pos + m, &mc));
    k_pair_ids<<<grid_for(m), kBlock, 0, c->st>>>(m, mate, pos, ids);
    RICH_LAUNCH_CHECK();
    k_compose<<<grid_for(n), kBlock, 0, c->st>>>(n, ids, agg);
    RICH_LAUNCH_CHECK();
    *nc = mc;
    if (pass + 1 < passes) {  // the pair graph's matrix for the next pass
      Csr<double> Pp, Rp, AP, Ac;
      Pp.nrows = m;
      Pp.ncols = mc;
      Pp.nnz = m;
      RICH_CHECK(dalloc(&Pp.rowptr, (long long)m + 1));
      RICH_CHECK(dalloc(&Pp.col, m));
      RICH_CHECK(dalloc(&Pp.val, m));
      k_iota<<<grid_for((long long)m + 1), kBlock, 0, c->st>>>(m + 1, Pp.rowptr);
      RICH_LAUNCH_CHECK();
      RICH_CUDA(cudaMemcpyAsync(Pp.col, ids, sizeof(int) * (size_t)m, cudaMemcpyDeviceToDevice, c->st));
      k_fill<<<grid_for(m), kBlock, 0, c->st>>>(m, 1.0, Pp.val);
      RICH_LAUNCH_CHECK();
      RICH_CHECK(transpose(c, Pp, Rp));
      RICH_CHECK(spgemm_symbolic(c, Ak, Pp, AP));
      RICH_CHECK(spgemm_symbolic(c, Rp, AP, Ac));
      csr_free(Pp);
      csr_free(Rp);
      csr_free(AP);
      if (own) csr_free(Ak);
      Ak = Ac;
      own = true;
    }
    dfree(d);
    dfree(w);
    dfree(mate);
    dfree(cand);
    dfree(first);
    dfree(pos);
    dfree(ids);
  }
  if (own) csr_free(Ak);
  return RICH_OK;
}

static int coarsen(rich_ctx* c, int l, bool* stop) {
  Hierarchy& H = c->H;
  const rich_amg_opts& o = H.opts;
  Level& L = H.lv[l];
  int n = L.n;
  *stop = false;
  double* d = nullptr;
  int* cnt = nullptr;
  Csr<double> S;
  RICH_CHECK(dalloc(&d, n));
  RICH_CHECK(dalloc(&cnt, n));
  k_diag<<<grid_for(n), kBlock, 0, c->st>>>(n, L.A.rowptr, L.A.col, L.A.val, d);
  RICH_LAUNCH_CHECK();
  int rounds = 0;
  int nc = 0;
  int* aggid = nullptr;
  bool unassigned = false;
  if (o.aggregation == RICH_AGG_MATCHING) {
    RICH_CHECK(dalloc(&L.agg, n));
    RICH_CHECK(dalloc(&aggid, 1));
    RICH_CHECK(matching_aggregate(c, L.A, o.max_agg_size, L.agg, &nc, &rounds));
  } else {
    double theta_l = o.theta * std::ldexp(1.0, -l);
    double theta2 = theta_l * theta_l;
    RICH_CHECK(strength(c, L.A, d, theta2, nullptr, cnt, nullptr));
    RICH_CHECK(dalloc(&S.rowptr, (long long)n + 1));
    RICH_CHECK(scan_exclusive_int(c, cnt, S.rowptr, n));
    int snnz = 0;
    RICH_CHECK(read_dev_int(c, S.rowptr + n, &snnz));
    RICH_CHECK(dalloc(&S.col, snnz));
    RICH_CHECK(strength(c, L.A, d, theta2, S.rowptr, nullptr, S.col));
    // MIS-2
    uint64_t *t = nullptr, *m1 = nullptr;
    RICH_CHECK(dalloc(&t, n));
    RICH_CHECK(dalloc(&m1, n));
    k_mis_init<<<grid_for(n), kBlock, 0, c->st>>>(n, o.seed, S.rowptr, t);
    RICH_LAUNCH_CHECK();
    for (;;) {
      RICH_CUDA(cudaMemsetAsync(c->iflag, 0, sizeof(int), c->st));
      k_max_closed<<<grid_for(n), kBlock, 0, c->st>>>(n, S.rowptr, S.col, t, m1);
      RICH_LAUNCH_CHECK();
      k_mis_update<<<grid_for(n), kBlock, 0, c->st>>>(n, S.rowptr, S.col, m1, t, c->iflag);
      RICH_LAUNCH_CHECK();
      ++rounds;
      RICH_CUDA(cudaMemcpyAsync(c->hflag, c->iflag, sizeof(int), cudaMemcpyDeviceToHost, c->st));
      RICH_CUDA(cudaStreamSynchronize(c->st));
      if (!c->hflag[0]) break;
      if (rounds > 100000) return RICH_ELIMIT;  // a round always decides the largest undecided key
    }
    // aggregates
    int* isroot = cnt;
    int* p1root = nullptr;
    uint64_t* rv = m1;
    uint64_t* best = nullptr;
    RICH_CHECK(dalloc(&aggid, (long long)n + 1));
    RICH_CHECK(dalloc(&p1root, n));
    RICH_CHECK(dalloc(&best, n));
    RICH_CHECK(dalloc(&L.agg, n));
    k_is_root<<<grid_for(n), kBlock, 0, c->st>>>(n, t, isroot);
    RICH_LAUNCH_CHECK();
    RICH_CHECK(scan_exclusive_int(c, isroot, aggid, n));
    RICH_CHECK(read_dev_int(c, aggid + n, &nc));
    k_rootval<<<grid_for(n), kBlock, 0, c->st>>>(n, t, rv);
    RICH_LAUNCH_CHECK();
    k_max_closed<<<grid_for(n), kBlock, 0, c->st>>>(n, S.rowptr, S.col, rv, best);
    RICH_LAUNCH_CHECK();
    k_agg_pass1<<<grid_for(n), kBlock, 0, c->st>>>(n, t, best, aggid, L.agg, p1root);
    RICH_LAUNCH_CHECK();
    k_val2<<<grid_for(n), kBlock, 0, c->st>>>(n, t, p1root, rv);
    RICH_LAUNCH_CHECK();
    k_max_closed<<<grid_for(n), kBlock, 0, c->st>>>(n, S.rowptr, S.col, rv, best);
    RICH_LAUNCH_CHECK();
    RICH_CUDA(cudaMemsetAsync(c->iflag, 0, sizeof(int), c->st));
    k_agg_pass2<<<grid_for(n), kBlock, 0, c->st>>>(n, S.rowptr, best, aggid, L.agg, c->iflag);
    RICH_LAUNCH_CHECK();
    RICH_CUDA(cudaMemcpyAsync(c->hflag, c->iflag, sizeof(int), cudaMemcpyDeviceToHost, c->st));
    RICH_CUDA(cudaStreamSynchronize(c->st));
    unassigned = c->hflag[0] != 0;
    if (!unassigned && o.isolated_join) {
      int* agg_in = p1root;  // pass-1 scratch, free now
      RICH_CUDA(cudaMemcpyAsync(agg_in, L.agg, sizeof(int) * (size_t)n, cudaMemcpyDeviceToDevice, c->st));
      k_agg_pass3<<<grid_for(n), kBlock, 0, c->st>>>(n, L.A.rowptr, L.A.col, L.A.val, o.seed, agg_in, L.agg);
      RICH_LAUNCH_CHECK();
    }
    dfree(t);
    dfree(m1);
    dfree(p1root);
    dfree(best);
    csr_free(S);
  }
  if (unassigned) {
    dfree(d);
    dfree(cnt);
    dfree(aggid);
    return RICH_ELIMIT;
  }
  L.mis_rounds = rounds;
  if (nc > 0.8 * n || nc < 1) {  // coarsening stalled: this level becomes the coarsest
    dfree(L.agg);
    dfree(d);
    dfree(cnt);
    dfree(aggid);
    *stop = true;
    return RICH_OK;
  }
  // prolongator: smoothed on the first smooth_levels levels, P_tent below
  Csr<double> Pt;
  Pt.nrows = n;
  Pt.ncols = nc;
  RICH_CHECK(dalloc(&Pt.rowptr, (long long)n + 1));
  k_ptent_count<<<grid_for(n), kBlock, 0, c->st>>>(n, L.agg, cnt);
  RICH_LAUNCH_CHECK();
  RICH_CHECK(scan_exclusive_int(c, cnt, Pt.rowptr, n));
  int ptnnz = 0;
  RICH_CHECK(read_dev_int(c, Pt.rowptr + n, &ptnnz));
  Pt.nnz = ptnnz;
  RICH_CHECK(dalloc(&Pt.col, ptnnz));
  k_ptent_fill<<<grid_for(n), kBlock, 0, c->st>>>(n, L.agg, Pt.rowptr, Pt.col);
  RICH_LAUNCH_CHECK();
  Pt.val = nullptr;
  if (l < o.smooth_levels) {
    int nb = red_grid(n);
    k_rowratio<<<nb, kBlock, 0, c->st>>>(n, L.A.rowptr, L.A.val, d, c->partials);
    RICH_LAUNCH_CHECK();
    RICH_CHECK(finish_max(c, c->partials, nb, c->dsc));
    double rho = 0.0;
    RICH_CHECK(fetch_scalars(c, c->dsc, 1, &rho));
    double omega = 4.0 / (3.0 * rho);
    L.omega = omega;
    Csr<double> Sm;
    Sm.nrows = Sm.ncols = n;
    Sm.nnz = L.A.nnz;
    Sm.rowptr = L.A.rowptr;
    Sm.col = L.A.col;
    RICH_CHECK(dalloc(&Sm.val, L.A.nnz));
    k_smoother_vals<<<grid_for(n), kBlock, 0, c->st>>>(n, L.A.rowptr, L.A.col, L.A.val, d, omega, Sm.val);
    RICH_LAUNCH_CHECK();
    RICH_CHECK(spgemm_symbolic(c, Sm, Pt, L.P));
    dfree(Sm.val);
  } else {
    // P = P_tent (pattern and unit values copied)
    L.omega = 0.0;
    L.P.nrows = n;
    L.P.ncols = nc;
    L.P.nnz = ptnnz;
    RICH_CHECK(dalloc(&L.P.rowptr, (long long)n + 1));
    RICH_CHECK(dalloc(&L.P.col, ptnnz));
    RICH_CHECK(dalloc(&L.P.val, ptnnz));
    RICH_CUDA(cudaMemcpyAsync(L.P.rowptr, Pt.rowptr, sizeof(int) * ((size_t)n + 1), cudaMemcpyDeviceToDevice, c->st));
    RICH_CUDA(cudaMemcpyAsync(L.P.col, Pt.col, sizeof(int) * (size_t)ptnnz, cudaMemcpyDeviceToDevice, c->st));
    k_fill<<<grid_for(ptnnz), kBlock, 0, c->st>>>(ptnnz, 1.0, L.P.val);
    RICH_LAUNCH_CHECK();
  }
  dfree(Pt.rowptr);
  dfree(Pt.col);
  RICH_CHECK(transpose(c, L.P, L.R));
  bool hashed_ap = false, hashed_rap = false;
  RICH_CHECK(spgemm_symbolic(c, L.A, L.P, L.AP, &L.u_ap, &hashed_ap));
  Level nxt;
  nxt.n = nc;
  RICH_CHECK(spgemm_symbolic(c, L.R, L.AP, nxt.A, &L.u_rap, &hashed_rap));
  if ((hashed_ap || hashed_rap) && o.product_lists) {
    // The next level's P is smoothed from these values and kept through every
    // refresh: sum them in the product lists' fixed order now (the lists the first
    // refresh would build), so that a setup does not depend on the order of atomics.
    L.pl_tried = true;
    RICH_CHECK(plist_build(c, L.A, L.P, L.AP, L.u_ap, L.pl_ap));
    if (L.pl_ap.built()) RICH_CHECK(plist_build(c, L.R, L.AP, nxt.A, L.u_rap, L.pl_rap));
    if (L.pl_ap.built() && L.pl_rap.built()) {
      RICH_CHECK(spgemm_numeric(c, L.A, L.P, L.AP, L.u_ap, 0, l, &L.pl_ap));
      RICH_CHECK(spgemm_numeric(c, L.R, L.AP, nxt.A, L.u_rap, 1, l, &L.pl_rap));
    }
  }
  if (c->prec == RICH_PREC_MIXED) {
    RICH_CHECK(dalloc(&L.P32, L.P.nnz));
    RICH_CHECK(dalloc(&L.R32, L.R.nnz));
    RICH_CHECK(dalloc(&L.AP32, L.AP.nnz));
    k_cast<<<grid_for(L.P.nnz), kBlock, 0, c->st>>>(L.P.nnz, L.P.val, L.P32);
    RICH_LAUNCH_CHECK();
    k_cast<<<grid_for(L.R.nnz), kBlock, 0, c->st>>>(L.R.nnz, L.R.val, L.R32);
    RICH_LAUNCH_CHECK();
  }
  dfree(d);
  dfree(cnt);
  dfree(aggid);
  H.lv.push_back(nxt);
  return RICH_OK;
}

int amg_build(rich_ctx* c, const rich_amg_opts* o) {
  if (!c->have_jac) return RICH_ESTATE;
  amg_free(c);
  Hierarchy& H = c->H;
  if (o) H.opts = *o; else rich_default_amg_opts(&H.opts);
  if (H.opts.max_levels < 1 || H.opts.max_levels > 16 || H.opts.nu1 < 0 || H.opts.nu2 < 0 || H.opts.coarse_max < 1)
    return RICH_EINVAL;
  if (H.opts.aggregation != RICH_AGG_MIS2 && H.opts.aggregation != RICH_AGG_MATCHING) return RICH_EINVAL;
  if (H.opts.smoother != RICH_SMOOTH_L1JACOBI && H.opts.smoother != RICH_SMOOTH_HYBRID_GS) return RICH_EINVAL;
  if (H.opts.smoother == RICH_SMOOTH_HYBRID_GS && (H.opts.hgs_seg < 1 || H.opts.hgs_block < 1 ||
                                                  H.opts.hgs_block > 4096))
    return RICH_EINVAL;
  if (H.opts.aggregation == RICH_AGG_MATCHING && (H.opts.max_agg_size < 2 || H.opts.max_agg_size > 1024))
    return RICH_EINVAL;
  if (H.opts.precond != RICH_PRECOND_AMG && H.opts.precond != RICH_PRECOND_AS) return RICH_EINVAL;
  if (H.opts.csr_layout < RICH_LAYOUT_AUTO || H.opts.csr_layout > RICH_LAYOUT_SELLP) return RICH_EINVAL;
  if (H.opts.graph != 0 && H.opts.graph != 1) return RICH_EINVAL;
  if (H.opts.precond == RICH_PRECOND_AS) {  // one level: the subdomain factors of A_aux
    RICH_CHECK(fine_stencil(c));
    RICH_CHECK(as_setup(c));
    H.built = true;
    return RICH_OK;
  }
  RICH_CHECK(refresh_a0_values(c));
  Level L0;
  L0.n = (int)c->g.n;
  L0.A = c->A0;  // aliases the context's finest CSR
  H.lv.push_back(L0);
  for (;;) {
    int l = (int)H.lv.size() - 1;
    if (H.lv[l].n < H.opts.coarse_max || (int)H.lv.size() >= H.opts.max_levels) break;
    bool stop = false;
    RICH_CHECK(coarsen(c, l, &stop));
    if (stop) break;
  }
  H.nlev = (int)H.lv.size();
  H.cn = H.lv[H.nlev - 1].n;
  // coarsening stalled above the dense limit: the coarsest level is smoothed
  H.dense = H.cn <= kMaxCoarseDense;
  H.scaled = H.nlev > 1 && H.opts.smoother == RICH_SMOOTH_L1JACOBI;
  for (int l = 0; l < H.nlev; ++l) {
    RICH_CHECK(level_alloc_vectors(c, H.lv[l]));
    RICH_CHECK(level_diag_data(c, H.lv[l], l > 0 || !H.scaled));
  }
  RICH_CHECK(fine_stencil(c));
  if (H.dense) {
    RICH_CHECK(dalloc(&H.cdense, (long long)H.cn * H.cn));
    RICH_CHECK(dalloc(&H.cwork, 2LL * kGjB * H.cn + kGjB * kGjB));
    if (c->prec == RICH_PREC_MIXED) RICH_CHECK(dalloc(&H.cinv32, (long long)H.cn * H.cn));
    RICH_CHECK(coarse_inverse(c));
    RICH_CHECK(capture_coarse_graph(c));
  }
  RICH_CUDA(cudaStreamSynchronize(c->st));
  H.built = true;
  return RICH_OK;
}

// New finest matrix: recompute every Galerkin product on the kept patterns.
int amg_refresh(rich_ctx* c) {
  Hierarchy& H = c->H;
  if (!H.built) return RICH_ESTATE;
  if (H.opts.precond == RICH_PRECOND_AS) {
    RICH_CHECK(fine_stencil(c));
    return as_setup(c);
  }
  RICH_CHECK(refresh_a0_values(c));
  H.lv[0].A = c->A0;
  for (int l = 0; l + 1 < H.nlev; ++l) {
    Level& L = H.lv[l];
    if (L.pl_tried || !H.opts.product_lists) continue;
    L.pl_tried = true;
    RICH_CHECK(plist_build(c, L.A, L.P, L.AP, L.u_ap, L.pl_ap));
    if (L.pl_ap.built()) RICH_CHECK(plist_build(c, L.R, L.AP, H.lv[l + 1].A, L.u_rap, L.pl_rap));
  }
  if (c->prec == RICH_PREC_MIXED) {
    // The V-cycle runs in FP32, so the Galerkin products do too: A32_{l+1} =
    // R32 (A32_l P32), on the patterns kept from the setup.  The FP64 values of
    // the coarse levels keep their setup-time content and are not read again.
    RICH_CHECK(level_diag_data(c, H.lv[0], !H.scaled));
    for (int l = 0; l + 1 < H.nlev; ++l) {
      Level& L = H.lv[l];
      Level& N = H.lv[l + 1];
      RICH_CHECK(spgemm_numeric_t<float>(c, L.A, L.A32, L.P, L.P32, L.AP, L.AP32, L.u_ap, 0, l, &L.pl_ap));
      RICH_CHECK(spgemm_numeric_t<float>(c, L.R, L.R32, L.AP, L.AP32, N.A, N.A32, L.u_rap, 1, l, &L.pl_rap));
      k_l1dinv32<<<grid_for(N.n), kBlock, 0, c->st>>>(N.n, N.A.rowptr, N.A32, N.dinv32);
      RICH_LAUNCH_CHECK();
    }
  } else {
    for (int l = 0; l + 1 < H.nlev; ++l) {
      Level& L = H.lv[l];
      RICH_CHECK(spgemm_numeric(c, L.A, L.P, L.AP, L.u_ap, 0, l, &L.pl_ap));
      RICH_CHECK(spgemm_numeric(c, L.R, L.AP, H.lv[l + 1].A, L.u_rap, 1, l, &L.pl_rap));
    }
    for (int l = H.scaled ? 1 : 0; l < H.nlev; ++l) RICH_CHECK(level_diag_data(c, H.lv[l]));
  }
  for (int l = 1; l < H.nlev; ++l) RICH_CHECK(sell_fill_a(c, H.lv[l]));
  RICH_CHECK(fine_stencil(c));
  return coarse_inverse(c);
}

// The paper's reuse: only the finest matrix and its smoother change.
int amg_update_fine(rich_ctx* c) {
  Hierarchy& H = c->H;
  if (!H.built) return RICH_ESTATE;
  if (H.opts.precond == RICH_PRECOND_AS) {
    RICH_CHECK(fine_stencil(c));
    return as_setup(c);
  }
  RICH_CHECK(refresh_a0_values(c));
  H.lv[0].A = c->A0;
  RICH_CHECK(level_diag_data(c, H.lv[0], !H.scaled, !H.scaled));
  RICH_CHECK(fine_stencil(c));
  if (H.nlev == 1) return coarse_inverse(c);
  return RICH_OK;
}

}  // namespace rich

using namespace rich;

extern "C" {

int amg_setup(rich_ctx* c, const rich_amg_opts* o, rich_amg_info* info) {
  if (!c) return RICH_EINVAL;
  AllocStream guard(c->st);
  RICH_CHECK(amg_build(c, o));
  if (info) {
    Hierarchy& H = c->H;
    memset(info, 0, sizeof(*info));
    if (H.opts.precond == RICH_PRECOND_AS || H.nlev == 0) return RICH_OK;  // no hierarchy: all zero
    info->levels = H.nlev;
    long long tot = 0;
    for (int l = 0; l < H.nlev && l < 16; ++l) {
      info->n[l] = H.lv[l].n;
      info->nnz[l] = H.lv[l].A.nnz;
      info->mis_rounds[l] = H.lv[l].mis_rounds;
      info->omega[l] = H.lv[l].omega;
      tot += H.lv[l].A.nnz;
    }
    info->operator_complexity = (double)tot / (double)H.lv[0].A.nnz;
  }
  return RICH_OK;
}

int amg_update(rich_ctx* c, int policy) {
  if (!c) return RICH_EINVAL;
  AllocStream guard(c->st);
  if (policy == RICH_AMG_SETUP_ONCE) return amg_update_fine(c);
  if (policy == RICH_AMG_REFRESH) return amg_refresh(c);
  return RICH_EINVAL;
}

int amg_export_level(rich_ctx* c, int level, int* agg, int* rp, int* col, double* val) {
  if (!c) return RICH_EINVAL;
  AllocStream guard(c->st);
  Hierarchy& H = c->H;
  if (!H.built) return RICH_ESTATE;
  if (level < 0 || level >= H.nlev) return RICH_EINVAL;
  Level& L = H.lv[level];
  RICH_CUDA(cudaStreamSynchronize(c->st));
  if (agg) {
    if (!L.agg) return RICH_EINVAL;
    RICH_CUDA(cudaMemcpy(agg, L.agg, sizeof(int) * L.n, cudaMemcpyDeviceToHost));
  }
  if (rp) RICH_CUDA(cudaMemcpy(rp, L.A.rowptr, sizeof(int) * (L.n + 1), cudaMemcpyDeviceToHost));
  if (col) RICH_CUDA(cudaMemcpy(col, L.A.col, sizeof(int) * L.A.nnz, cudaMemcpyDeviceToHost));
  if (val) {
    if (c->prec == RICH_PREC_MIXED && level > 0) {
      // the FP32 values the V-cycle uses (refreshed in FP32), widened
      std::vector<float> v32((size_t)L.A.nnz);
      RICH_CUDA(cudaMemcpy(v32.data(), L.A32, sizeof(float) * L.A.nnz, cudaMemcpyDeviceToHost));
      for (long long e = 0; e < L.A.nnz; ++e) val[e] = (double)v32[(size_t)e];
    } else {
      RICH_CUDA(cudaMemcpy(val, L.A.val, sizeof(double) * L.A.nnz, cudaMemcpyDeviceToHost));
    }
  }
  return RICH_OK;
}

int amg_export_prolongator(rich_ctx* c, int level, long long* nnz, int* rp, int* col, double* val) {
  if (!c) return RICH_EINVAL;
  AllocStream guard(c->st);
  Hierarchy& H = c->H;
  if (!H.built) return RICH_ESTATE;
  if (level < 0 || level + 1 >= H.nlev) return RICH_EINVAL;
  Level& L = H.lv[level];
  RICH_CUDA(cudaStreamSynchronize(c->st));
  if (nnz) *nnz = L.P.nnz;
  if (rp) RICH_CUDA(cudaMemcpy(rp, L.P.rowptr, sizeof(int) * (L.n + 1), cudaMemcpyDeviceToHost));
  if (col) RICH_CUDA(cudaMemcpy(col, L.P.col, sizeof(int) * L.P.nnz, cudaMemcpyDeviceToHost));
  if (val) RICH_CUDA(cudaMemcpy(val, L.P.val, sizeof(double) * L.P.nnz, cudaMemcpyDeviceToHost));
  return RICH_OK;
}

}  // extern "C"

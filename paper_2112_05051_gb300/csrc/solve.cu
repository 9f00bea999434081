// V-cycle (eq. (Vcycle), Sec. 5.2), flexible Krylov solvers for the right-
// preconditioned Newton system (eq. (precsystem), Sec. 3) and the inexact
// Newton-Armijo backward-Euler step (Sec. 3).
//
// V-cycle on level l with zero initial guess: nu1 l1-Jacobi sweeps
// x <- x + D_l1^-1 (b - A x), residual r = b - A x, b_{l+1} = R r, recursion
// (the coarsest level multiplies by its dense inverse), x <- x + P x_{l+1},
// nu2 sweeps.  In MIXED precision every level works in FP32 with FP32
// accumulation; the Krylov vectors and dot products stay FP64.
//
// Krylov scalars live in device memory.  FGMRES reads one small block of them back per
// iteration for the convergence test; FCG tests on the device and is read when it stops.
#include <algorithm>
#include <cstdio>
#include <map>
#include <mutex>
#include <vector>

#include "gram.cuh"

namespace rich {

// ---------------------------------------------------------------- V-cycle kernels (T = double | float)

template <class T>
__global__ void k_jacobi0(int n, const T* __restrict__ dinv, const T* __restrict__ b, T* __restrict__ x) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) x[i] = dinv[i] * b[i];
}

// CSR row operation with G lanes per row (G = 1..32), for levels whose rows are
// long (coarse Galerkin operators carry tens to hundreds of entries per row).
// MODE 0: y = A x, and y2 = dinv y if y2 (a level's right-hand side and its first sweep);
// 1: y += A x; 2: y = x + dinv (b - A x); 3: y = b - A x; 4: y = b + dinv (A x).
// U = 4: a lane takes entries e, e+G, e+2G, e+3G at a time, absent ones predicated off, so
// that a batch costs one round of loads (columns and values, then the gathers) whatever
// the row's length, and the row's own operands are in flight meanwhile; the coarse levels
// are bound by that latency (8876 rows of 101 entries, FP64: 9.1 us in rounds of one).
template <class T, int MODE, int G, int U = 1>
__global__ void k_csr_grp(int n, const int* __restrict__ rp, const int* __restrict__ col, const T* __restrict__ val,
                          const T* __restrict__ dinv, const T* __restrict__ b, const T* __restrict__ x,
                          T* __restrict__ y, T* __restrict__ y2) {
  int lane = threadIdx.x & (G - 1);
  unsigned mask = G == 32 ? 0xffffffffu : (((1u << G) - 1) << ((threadIdx.x & 31) & ~(G - 1)));
  int rows_per_grid = (gridDim.x * blockDim.x) / G;
  for (int row = (blockIdx.x * blockDim.x + threadIdx.x) / G; row < n; row += rows_per_grid) {
    T s = 0;
    int e = rp[row] + lane;
    const int end = rp[row + 1];
    T bi = 0, xi = 0, di = 0;  // the row's own operands
    if (lane == 0) {
      if (MODE >= 2) bi = b[row];
      if (MODE == 2) xi = x[row];
      if (MODE == 1) xi = y[row];
      if (MODE == 2 || MODE == 4 || (MODE == 0 && y2)) di = dinv[row];
    }
    if (U == 4) {
      T s1 = 0;
      for (; e < end; e += 4 * G) {
        int c[4];
        T v[4], xx[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const bool in = e + u * G < end;
          c[u] = in ? col[e + u * G] : -1;
          v[u] = in ? val[e + u * G] : T(0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) xx[u] = c[u] >= 0 ? x[c[u]] : T(0);
        s += v[0] * xx[0];
        s1 += v[1] * xx[1];
        s += v[2] * xx[2];
        s1 += v[3] * xx[3];
      }
      s += s1;
    } else {
      for (; e < end; e += G) s += val[e] * x[col[e]];
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) s += __shfl_down_sync(mask, s, o, G);
    if (lane == 0) {
      if (MODE == 0) {
        y[row] = s;
        if (y2) y2[row] = di * s;
      } else if (MODE == 1) y[row] = xi + s;
      else if (MODE == 2) y[row] = xi + di * (bi - s);
      else if (MODE == 3) y[row] = bi - s;
      else y[row] = bi + di * s;
    }
  }
}

// The same row operations on the SELL-C-sigma copy: one warp per slice of 32 rows,
// one thread per row, slot loads coalesced across the warp, U gathers of x in flight
// per thread (U = 4 or 8), no cross-lane reduction (on GB300's narrow FP64 pipe the
// shuffle-add reductions and the idle lanes of ragged rows cost as much as the
// products themselves).  Past a row's end the slots hold zeros.
template <class T, int MODE, int U>
__global__ void __launch_bounds__(U == 4 ? kSellSigma : kBlock) k_sell(int nslice, const int* __restrict__ sptr,
                                                 const int* __restrict__ perm, const int* __restrict__ col,
                                                 const T* __restrict__ val, const T* __restrict__ dinv,
                                                 const T* __restrict__ b, const T* __restrict__ x,
                                                 T* __restrict__ y, T* __restrict__ y2) {
  const int lane = threadIdx.x & (kSellC - 1);
  const int warps = (gridDim.x * blockDim.x) / kSellC;
  for (int s = (blockIdx.x * blockDim.x + threadIdx.x) / kSellC; s < nslice; s += warps) {
    const int row = perm[s * kSellC + lane];
    const int end = sptr[s + 1];
    int e = sptr[s] + lane;
    T s0 = 0, s1 = 0;
    for (; e + (U - 1) * kSellC < end; e += U * kSellC) {  // warp-uniform: the slice's columns are full
      int cc[U];
      T vv[U], xx[U];
#pragma unroll
      for (int u = 0; u < U; ++u) cc[u] = col[e + u * kSellC];
#pragma unroll
      for (int u = 0; u < U; ++u) vv[u] = val[e + u * kSellC];
#pragma unroll
      for (int u = 0; u < U; ++u) xx[u] = x[cc[u]];
#pragma unroll
      for (int u = 0; u < U; u += 2) {
        s0 += vv[u] * xx[u];
        s1 += vv[u + 1] * xx[u + 1];
      }
    }
    if (U == 8) {  // (the batched form below takes 64 registers here and costs 2 us of 21)
      for (; e < end; e += kSellC) s0 += val[e] * x[col[e]];
    } else {  // the last columns, one round of loads for all of them (warp-uniform tests)
      const int rem = (end - e + lane) / kSellC;
      int cc[U - 1];
      T vv[U - 1], xx[U - 1];
#pragma unroll
      for (int u = 0; u < U - 1; ++u)
        if (u < rem) {
          cc[u] = col[e + u * kSellC];
          vv[u] = val[e + u * kSellC];
        }
#pragma unroll
      for (int u = 0; u < U - 1; ++u)
        if (u < rem) xx[u] = x[cc[u]];
#pragma unroll
      for (int u = 0; u < U - 1; ++u)
        if (u < rem) s0 += vv[u] * xx[u];
    }
    const T a = s0 + s1;
    if (row >= 0) {
      if (MODE == 0) {
        y[row] = a;
        if (y2) y2[row] = dinv[row] * a;
      } else if (MODE == 1) y[row] += a;
      else if (MODE == 2) y[row] = x[row] + dinv[row] * (b[row] - a);
      else if (MODE == 3) y[row] = b[row] - a;
      else y[row] = b[row] + dinv[row] * a;
    }
  }
}

// SELL, software-pipelined: while the gathers of x for four columns and their
// products run, the slot loads (column and value) of the next four are already in
// flight, so the DRAM latency of the copy overlaps the L2 latency of the gathers
// instead of adding to it.
template <class T, int MODE>
__global__ void __launch_bounds__(kBlock) k_sellp(int nslice, const int* __restrict__ sptr,
                                                  const int* __restrict__ perm, const int* __restrict__ col,
                                                  const T* __restrict__ val, const T* __restrict__ dinv,
                                                  const T* __restrict__ b, const T* __restrict__ x,
                                                  T* __restrict__ y, T* __restrict__ y2) {
  const int lane = threadIdx.x & (kSellC - 1);
  const int warps = (gridDim.x * blockDim.x) / kSellC;
  for (int s = (blockIdx.x * blockDim.x + threadIdx.x) / kSellC; s < nslice; s += warps) {
    const int row = perm[s * kSellC + lane];
    const int end = sptr[s + 1];
    int e = sptr[s] + lane;
    T s0 = 0, s1 = 0;
    bool have = e + 3 * kSellC < end;  // warp-uniform, as every test below
    int c0 = 0, c1 = 0, c2 = 0, c3 = 0;
    T v0 = 0, v1 = 0, v2 = 0, v3 = 0;
    if (have) {
      c0 = col[e];
      c1 = col[e + kSellC];
      c2 = col[e + 2 * kSellC];
      c3 = col[e + 3 * kSellC];
      v0 = val[e];
      v1 = val[e + kSellC];
      v2 = val[e + 2 * kSellC];
      v3 = val[e + 3 * kSellC];
    }
    while (have) {
      const int en = e + 4 * kSellC;
      const bool next = en + 3 * kSellC < end;
      int d0 = 0, d1 = 0, d2 = 0, d3 = 0;
      T w0 = 0, w1 = 0, w2 = 0, w3 = 0;
      if (next) {
        d0 = col[en];
        d1 = col[en + kSellC];
        d2 = col[en + 2 * kSellC];
        d3 = col[en + 3 * kSellC];
        w0 = val[en];
        w1 = val[en + kSellC];
        w2 = val[en + 2 * kSellC];
        w3 = val[en + 3 * kSellC];
      }
      const T x0 = x[c0], x1 = x[c1], x2 = x[c2], x3 = x[c3];
      s0 += v0 * x0;
      s1 += v1 * x1;
      s0 += v2 * x2;
      s1 += v3 * x3;
      c0 = d0;
      c1 = d1;
      c2 = d2;
      c3 = d3;
      v0 = w0;
      v1 = w1;
      v2 = w2;
      v3 = w3;
      e = en;
      have = next;
    }
    for (; e < end; e += kSellC) s0 += val[e] * x[col[e]];
    const T a = s0 + s1;
    if (row >= 0) {
      if (MODE == 0) {
        y[row] = a;
        if (y2) y2[row] = dinv[row] * a;
      } else if (MODE == 1) y[row] += a;
      else if (MODE == 2) y[row] = x[row] + dinv[row] * (b[row] - a);
      else if (MODE == 3) y[row] = b[row] - a;
      else y[row] = b[row] + dinv[row] * a;
    }
  }
}

// SELL with two lanes per row: one warp per half-slice (16 rows); lane t + 16 ph
// takes the row's columns j = ph, ph + 2, ... (each load instruction reads two
// contiguous 128-byte runs), and one shuffle-add joins the two partial sums.  Twice
// the warps of k_sell for the same slices: more loads in flight on levels whose
// slices alone fill only part of the GPU.
template <class T, int MODE>
__global__ void __launch_bounds__(kBlock) k_sell2(int nslice, const int* __restrict__ sptr,
                                                  const int* __restrict__ perm, const int* __restrict__ col,
                                                  const T* __restrict__ val, const T* __restrict__ dinv,
                                                  const T* __restrict__ b, const T* __restrict__ x,
                                                  T* __restrict__ y, T* __restrict__ y2) {
  const int lane = threadIdx.x & 31, ph = lane >> 4;
  const int warps = (gridDim.x * blockDim.x) / 32;
  for (int hs = (blockIdx.x * blockDim.x + threadIdx.x) / 32; hs < 2 * nslice; hs += warps) {
    const int s = hs >> 1, r = (hs & 1) * 16 + (lane & 15);
    const int row = perm[s * kSellC + r];
    const int base = sptr[s] + r, w = (sptr[s + 1] - sptr[s]) / kSellC;
    T s0 = 0, s1 = 0;
    int j = ph;
    for (; j + 6 < w; j += 8) {  // columns j, j + 2, j + 4, j + 6 of this lane
      const int c0 = col[base + j * kSellC], c1 = col[base + (j + 2) * kSellC];
      const int c2 = col[base + (j + 4) * kSellC], c3 = col[base + (j + 6) * kSellC];
      const T v0 = val[base + j * kSellC], v1 = val[base + (j + 2) * kSellC];
      const T v2 = val[base + (j + 4) * kSellC], v3 = val[base + (j + 6) * kSellC];
      const T x0 = x[c0], x1 = x[c1], x2 = x[c2], x3 = x[c3];
      s0 += v0 * x0;
      s1 += v1 * x1;
      s0 += v2 * x2;
      s1 += v3 * x3;
    }
    for (; j < w; j += 2) s0 += val[base + j * kSellC] * x[col[base + j * kSellC]];
    T a = s0 + s1;
    a += __shfl_xor_sync(0xffffffffu, a, 16);
    if (ph == 0 && row >= 0) {
      if (MODE == 0) {
        y[row] = a;
        if (y2) y2[row] = dinv[row] * a;
      } else if (MODE == 1) y[row] += a;
      else if (MODE == 2) y[row] = x[row] + dinv[row] * (b[row] - a);
      else if (MODE == 3) y[row] = b[row] - a;
      else y[row] = b[row] + dinv[row] * a;
    }
  }
}

// Variant v of the CSR row kernel: lanes per row G = v & 0xff, four-way unrolled
// rows when v & kUnroll; v == kSellVariant (4 gathers in flight per thread),
// kSellVariant8 (8), kSellVariant2 (two lanes per row) or kSellVariantP
// (software-pipelined) runs the SELL copy (sl, sval) instead.
constexpr int kUnroll = 0x100;
constexpr int kSellVariant = 0x200;
constexpr int kSellVariant8 = 0x201;
constexpr int kSellVariant2 = 0x202;
constexpr int kSellVariantP = 0x203;
inline bool is_sell(int v) { return (v & kSellVariant) != 0; }
template <class T, int MODE>
static void csr_launch(cudaStream_t st, int v, int n, const int* rp, const int* col, const T* val, const T* dinv,
                       const T* b, const T* x, T* y, const Sell* sl = nullptr, const T* sval = nullptr,
                       T* y2 = nullptr) {
  if (is_sell(v)) {
    const int g = grid_for((long long)sl->nslice * kSellC);
    // a block per window of the sort: its vectors' accesses, in sorted order, share L1 lines
    const int gw = grid_for((long long)sl->nslice * kSellC, kSellSigma);
    if (v == kSellVariant8)
      k_sell<T, MODE, 8><<<g, kBlock, 0, st>>>(sl->nslice, sl->sptr, sl->perm, sl->col, sval, dinv, b, x, y, y2);
    else if (v == kSellVariant2)
      k_sell2<T, MODE><<<grid_for(2LL * sl->nslice * kSellC), kBlock, 0, st>>>(sl->nslice, sl->sptr, sl->perm,
                                                                               sl->col, sval, dinv, b, x, y, y2);
    else if (v == kSellVariantP)
      k_sellp<T, MODE><<<g, kBlock, 0, st>>>(sl->nslice, sl->sptr, sl->perm, sl->col, sval, dinv, b, x, y, y2);
    else
      k_sell<T, MODE, 4><<<gw, kSellSigma, 0, st>>>(sl->nslice, sl->sptr, sl->perm, sl->col, sval, dinv, b, x, y, y2);
    return;
  }
  const int G = v & 0xff;
  long long thr = (long long)n * G;
  const dim3 gr(grid_for(thr));
  if (v & kUnroll) {
    switch (G) {
      case 1: k_csr_grp<T, MODE, 1, 4><<<gr, kBlock, 0, st>>>(n, rp, col, val, dinv, b, x, y, y2); break;
      case 2: k_csr_grp<T, MODE, 2, 4><<<gr, kBlock, 0, st>>>(n, rp, col, val, dinv, b, x, y, y2); break;
      case 4: k_csr_grp<T, MODE, 4, 4><<<gr, kBlock, 0, st>>>(n, rp, col, val, dinv, b, x, y, y2); break;
      case 8: k_csr_grp<T, MODE, 8, 4><<<gr, kBlock, 0, st>>>(n, rp, col, val, dinv, b, x, y, y2); break;
      case 16: k_csr_grp<T, MODE, 16, 4><<<gr, kBlock, 0, st>>>(n, rp, col, val, dinv, b, x, y, y2); break;
      default: k_csr_grp<T, MODE, 32, 4><<<gr, kBlock, 0, st>>>(n, rp, col, val, dinv, b, x, y, y2); break;
    }
    return;
  }
  switch (G) {
    case 1: k_csr_grp<T, MODE, 1><<<gr, kBlock, 0, st>>>(n, rp, col, val, dinv, b, x, y, y2); break;
    case 2: k_csr_grp<T, MODE, 2><<<gr, kBlock, 0, st>>>(n, rp, col, val, dinv, b, x, y, y2); break;
    case 4: k_csr_grp<T, MODE, 4><<<gr, kBlock, 0, st>>>(n, rp, col, val, dinv, b, x, y, y2); break;
    case 8: k_csr_grp<T, MODE, 8><<<gr, kBlock, 0, st>>>(n, rp, col, val, dinv, b, x, y, y2); break;
    case 16: k_csr_grp<T, MODE, 16><<<gr, kBlock, 0, st>>>(n, rp, col, val, dinv, b, x, y, y2); break;
    default: k_csr_grp<T, MODE, 32><<<gr, kBlock, 0, st>>>(n, rp, col, val, dinv, b, x, y, y2); break;
  }
}

// Lanes per row when nothing has been measured: one thread per short row, wider
// groups as rows grow.
static int default_lanes(double avg) {
  if (avg <= 6) return 1;
  if (avg > 96) return 32;
  if (avg > 64) return 16;
  if (avg > 40) return 8;
  return 4;
}

// Autotuner of the CSR row operations: the first time an operation meets a shape
// class (mode, value type, rows in quarter-octave bins, mean row length rounded to
// an integer), every candidate is timed on the actual operands (output to a scratch
// vector, two rounds behind a warm-up launch each, CUDA events) and the fastest
// is kept for the rest of the process.  Classes, not exact shapes, so that
// a stream of requests of similar size (whose coarse levels differ by a few rows)
// tunes once.  The table is shared by all contexts (under a mutex, held while
// tuning, so concurrent requests of one class agree); a class therefore always runs
// the same kernel, and results do not depend on what else is in flight.
struct TuneKey {
  int mode, tsize, n;   // n: quarter-octave bin of the row count
  long long nnz;        // rounded mean row length
  int sell;             // 1: a SELL copy is among the candidates
  bool operator<(const TuneKey& o) const {
    if (mode != o.mode) return mode < o.mode;
    if (tsize != o.tsize) return tsize < o.tsize;
    if (n != o.n) return n < o.n;
    if (nnz != o.nnz) return nnz < o.nnz;
    return sell < o.sell;
  }
};
struct TuneVal {
  int variant;   // fastest candidate
  float us;      // its time per launch
  int best_csr;  // fastest CSR candidate (used where a matrix of the class has no SELL copy)
};
constexpr long long kTuneDelay = 40000;  // ~20 us: the host gets ahead of the timed launches
constexpr size_t kTuneLast = 6;          // candidates of the second round at most
constexpr float kTuneTick = 2.1f;        // us: what the length of a timed run is rounded to
struct TuneEvents {
  std::vector<cudaEvent_t> e;
  bool ok = true;
  explicit TuneEvents(size_t n) : e(n, nullptr) {
    for (auto& x : e) ok = ok && cudaEventCreate(&x) == cudaSuccess;
  }
  ~TuneEvents() {
    for (auto x : e)
      if (x) cudaEventDestroy(x);
  }
};
static std::mutex g_tune_mu;
static std::map<TuneKey, TuneVal> g_tune;

// Where a row operation's matrix can get a SELL copy: the copy, the CSR it is laid
// out from and the values in the hierarchy precision.
template <class T>
struct SellSrc {
  Sell* s;
  const Csr<double>* M;
  const T* vals;
};

// Lays out the SELL copy on first use (the row operations of a class that chose it,
// or a class being tuned): matrices whose class keeps CSR never get one.
template <class T>
static int sell_ensure(rich_ctx* c, const SellSrc<T>& src, bool* ok) {
  if (!src.s->built()) {
    RICH_CHECK(sell_build(c, *src.M, *src.s));
    if (src.s->built()) RICH_CHECK(sell_fill(c, *src.M, src.vals, *src.s));
    prof_restart(c->st);
  }
  *ok = src.s->built();
  return RICH_OK;
}

// src: the matrix's SELL source (nullptr: CSR only).
template <class T, int MODE>
static int csr_op(rich_ctx* c, int n, long long nnz, const int* rp, const int* col, const T* val, const T* dinv,
                  const T* b, const T* x, T* y, const SellSrc<T>* src = nullptr, T* y2 = nullptr) {
  if (n <= 0) return RICH_OK;
  const int layout = c->H.opts.csr_layout;
  const bool offer = src && src->s && n >= kSellMinRows && layout != RICH_LAYOUT_CSR;
  int v = default_lanes((double)nnz / n);
  bool sell_ok = false;
  if (offer && layout >= RICH_LAYOUT_SELL) {  // a SELL kernel named by the option
    RICH_CHECK(sell_ensure(c, *src, &sell_ok));
    if (sell_ok)
      v = layout == RICH_LAYOUT_SELL8   ? kSellVariant8
          : layout == RICH_LAYOUT_SELL2 ? kSellVariant2
          : layout == RICH_LAYOUT_SELLP ? kSellVariantP
                                        : kSellVariant;
  } else if (c->H.opts.autotune) {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    TuneKey key{MODE, (int)sizeof(T), (int)std::floor(4.0 * std::log2((double)n)),
                (long long)std::llround((double)nnz / n), offer ? 1 : 0};
    auto it = g_tune.find(key);
    if (it != g_tune.end()) {
      v = it->second.variant;
      if (is_sell(v)) {
        RICH_CHECK(sell_ensure(c, *src, &sell_ok));
        if (!sell_ok) v = it->second.best_csr;
      }
    } else if (!profiling_active()) {  // a profiled pass runs what is tuned, and tunes nothing
      const bool had_copy = offer && src->s->built();
      if (offer) RICH_CHECK(sell_ensure(c, *src, &sell_ok));
      T* scratch = nullptr;
      RICH_CHECK(dalloc(&scratch, n));
      RICH_CUDA(cudaMemsetAsync(scratch, 0, sizeof(T) * (size_t)n, c->st));
      // Back-to-back launches on warm operands.  Timing each launch from a cold L2
      // (a 256 MB write before it) was measured and chose worse variants: the same
      // headline, 3 % less in the mixed mode, whose FP32 levels stay in L2 between
      // the sweeps of a V-cycle.
      float best = 1e30f, best_csr_us = 1e30f;
      int best_csr = v;
      const Sell* sl = sell_ok ? src->s : nullptr;
      const T* sval = sell_ok ? (sizeof(T) == 8 ? (const T*)sl->val : (const T*)sl->val32) : nullptr;
      // us per launch of each candidate: the launches queue up behind a delay, so that the
      // events see the GPU alone, and all are waited for once.
      auto measure = [&](const std::vector<int>& cand, const std::vector<int>& reps, std::vector<float>& us) -> int {
        TuneEvents ev(2 * cand.size());
        if (!ev.ok) return RICH_ECUDA;
        gpu_delay(c->st, kTuneDelay);
        for (size_t k = 0; k < cand.size(); ++k) {
          csr_launch<T, MODE>(c->st, cand[k], n, rp, col, val, dinv, b, x, scratch, sl, sval, y2);
          RICH_CUDA(cudaEventRecord(ev.e[2 * k], c->st));
          for (int rep = 0; rep < reps[k]; ++rep)
            csr_launch<T, MODE>(c->st, cand[k], n, rp, col, val, dinv, b, x, scratch, sl, sval, y2);
          RICH_CUDA(cudaEventRecord(ev.e[2 * k + 1], c->st));
          count_launches(1 + reps[k]);
        }
        RICH_CUDA(cudaEventSynchronize(ev.e.back()));
        us.resize(cand.size());
        for (size_t k = 0; k < cand.size(); ++k) {
          RICH_CUDA(cudaEventElapsedTime(&us[k], ev.e[2 * k], ev.e[2 * k + 1]));
          us[k] *= 1000.f / reps[k];
        }
        return RICH_OK;
      };
      // First two launches of each, then runs of about 60 us of those that two launches cannot
      // tell from the fastest.  (A first V-cycle, V(1,1) at 128^3 FP64, and the later ones: 50 ms
      // and 281 us with a wait, 30 us of delay and three launches per candidate; 45 ms and 290
      // with one wait for all, small kernels' ties being settled by their order; 36 ms and 281 so.)
      std::vector<int> cand;
      for (int g : {1, 2, 4, 8, 16, 32, 1 | kUnroll, 2 | kUnroll, 4 | kUnroll, 8 | kUnroll, 16 | kUnroll,
                    32 | kUnroll, kSellVariant, kSellVariant8, kSellVariant2, kSellVariantP})
        if (!is_sell(g) || sell_ok) cand.push_back(g);
      std::vector<float> us, us2;
      RICH_CHECK(measure(cand, std::vector<int>(cand.size(), 2), us));
      std::vector<size_t> by(cand.size());
      for (size_t k = 0; k < by.size(); ++k) by[k] = k;
      std::stable_sort(by.begin(), by.end(), [&](size_t p, size_t q) { return us[p] < us[q]; });
      std::vector<int> last, reps;
      for (size_t k : by) {
        if (last.size() == kTuneLast || us[k] > 1.02f * us[by[0]] + 0.5f * kTuneTick) break;
        last.push_back(cand[k]);
        reps.push_back(std::max(2, (int)std::min(12.f, 60.f / us[k])));
      }
      if (last.size() > 1) {
        RICH_CHECK(measure(last, reps, us2));
        for (size_t k = 0; k < last.size(); ++k) us[by[k]] = us2[k];
      }
      for (size_t k = 0; k < by.size(); ++k) {
        const int g = cand[by[k]];
        if (k < last.size() && us[by[k]] < best) {
          best = us[by[k]];
          v = g;
        }
        if (!is_sell(g) && us[by[k]] < best_csr_us) {
          best_csr_us = us[by[k]];
          best_csr = g;
        }
      }
      RICH_CUDA(cudaGetLastError());
      dfree(scratch);
      g_tune[key] = {v, best, best_csr};
      if (sell_ok && !is_sell(v) && !had_copy) {  // the copy lost: not kept, not refreshed
        sell_free(*src->s);
        sell_ok = false;
      }
    }
  }
  const Sell* sl = nullptr;
  const T* sval = nullptr;
  if (is_sell(v)) {
    sl = src->s;
    sval = sizeof(T) == 8 ? (const T*)sl->val : (const T*)sl->val32;
  }
  csr_launch<T, MODE>(c->st, v, n, rp, col, val, dinv, b, x, y, sl, sval, y2);
  return RICH_OK;
}

int autotune_table(char* buf, int cap) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  int off = 0;
  buf[0] = 0;
  for (auto& e : g_tune) {
    int w = snprintf(buf + off, cap - off, "%d %d %d %lld %d %d %.3f %d\n", e.first.mode, e.first.tsize,
                     e.first.n, e.first.nnz, e.first.sell, e.second.variant, e.second.us, e.second.best_csr);
    if (w < 0 || w >= cap - off) break;
    off += w;
  }
  return RICH_OK;
}

// Entries in autotune_table's format (a saved table): classes already present keep
// their choice.  A variant that is not one of the candidates is rejected.
int autotune_load(const char* text) {
  auto valid = [](int v) {
    if (v == kSellVariant || v == kSellVariant8 || v == kSellVariant2 || v == kSellVariantP) return true;
    const int g = v & 0xff, u = v & ~0xff;
    if (u != 0 && u != kUnroll) return false;
    return g == 1 || g == 2 || g == 4 || g == 8 || g == 16 || g == 32;
  };
  std::vector<std::pair<TuneKey, TuneVal>> rows;
  const char* p = text;
  while (*p) {
    int mode, tsize, n, sell, variant, best_csr, used = 0;
    long long nnz;
    float us;
    if (sscanf(p, "%d %d %d %lld %d %d %f %d%n", &mode, &tsize, &n, &nnz, &sell, &variant, &us, &best_csr, &used) !=
        8)
      return RICH_EINVAL;
    if (mode < 0 || mode > 4 || (tsize != 4 && tsize != 8) || (sell != 0 && sell != 1) || !valid(variant) ||
        !valid(best_csr) || best_csr >= kSellVariant || (!sell && variant >= kSellVariant))
      return RICH_EINVAL;
    rows.push_back({TuneKey{mode, tsize, n, nnz, sell}, TuneVal{variant, us, best_csr}});
    p += used;
    while (*p == '\n' || *p == ' ' || *p == '\r') ++p;
  }
  std::lock_guard<std::mutex> lk(g_tune_mu);
  for (auto& r : rows) g_tune.insert(r);
  return RICH_OK;
}

// x = M b for a dense row-major n x n matrix; one warp per row, 8 loads of either in
// flight per lane (n = 362 in FP64: 10 us with one at a time).
template <class T>
__global__ void k_gemv(int n, const T* __restrict__ M, const T* __restrict__ b, T* __restrict__ x) {
  int lane = threadIdx.x & 31;
  for (int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < n; row += (gridDim.x * blockDim.x) >> 5) {
    const T* m = M + (long long)row * n;
    T s = 0, s1 = 0;
    for (int j = lane; j < n; j += 256) {
      T a[8], v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const bool in = j + 32 * u < n;
        a[u] = in ? m[j + 32 * u] : T(0);
        v[u] = in ? b[j + 32 * u] : T(0);
      }
#pragma unroll
      for (int u = 0; u < 8; u += 2) {
        s += a[u] * v[u];
        s1 += a[u + 1] * v[u + 1];
      }
    }
    s += s1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) x[row] = s;
  }
}

__global__ void k_d2f(long long n, const double* __restrict__ a, float* __restrict__ b) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    b[i] = (float)a[i];
}
__global__ void k_f2d(long long n, const float* __restrict__ a, double* __restrict__ b) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    b[i] = (double)a[i];
}

// Finest-level residual xo = b - A x on the stencil form (hybrid Gauss-Seidel's).
template <class T>
__global__ void __launch_bounds__(kLineThreads) k_st_resid(GridP g, Stencil4<T> A, const T* __restrict__ b,
                                                            const T* __restrict__ x, T* __restrict__ xo) {
  int i = blockIdx.y * kLineThreads + threadIdx.x;
  if (i >= g.nx) return;
  int r = blockIdx.x;
  int j = r % g.ny;
  int k = r / g.ny;
  int nx = g.nx;
  int sxy = g.nx * g.ny;
  int c = r * nx + i;
  T wxp = A.wx[c], wyp = A.wy[c], wzp = A.wz[c];
  T xc = x[c];
  T ax = A.diag[c] * xc;
  if (i > 0) ax -= A.wx[c - 1] * x[c - 1];
  if (i < nx - 1) ax -= wxp * x[c + 1];
  if (j > 0) ax -= A.wy[c - nx] * x[c - nx];
  if (j < g.ny - 1) ax -= wyp * x[c + nx];
  if (k > 0) ax -= A.wz[c - sxy] * x[c - sxy];
  if (k < g.nz - 1) ax -= wzp * x[c + sxy];
  xo[c] = b[c] - ax;
}

// Sweep (MODE 1: out = b' + (I - A') y) and residual (MODE 2: out = q (b' - A' y), the
// unscaled residual, with A's own diagonal -gd) of the scaled finest level (ScaledSt).  A thread marches zc layers with
// its column's y and vertical weight in registers.
// Bound: FP64, one multiply-add per entry; FP32, HBM (28 bytes per cell: g, 3 weights, b, y
// in, y out).  128^3 FP64: the unscaled sweep, 9 operations and 64 bytes, took 36 us, and
// the first sweep from zero, a pass of its own (9 us), is gone.
template <class T, int MODE>
__global__ void __launch_bounds__(kLineThreads) k_sc(GridP g, ScaledSt<T> A, int zc, const T* __restrict__ b,
                                                     const T* __restrict__ y, T* __restrict__ out) {
  const int i = blockIdx.y * blockDim.x + threadIdx.x;
  if (i >= g.nx) return;
  const int j = blockIdx.x % g.ny, k0 = blockIdx.x / g.ny * zc, k1 = min(g.nz, k0 + zc);
  const int nx = g.nx, sxy = g.nx * g.ny;
  int c = (k0 * g.ny + j) * nx + i;
  T ym = T(0), wm = T(0), yc = y[c];
  if (k0 > 0) {
    ym = y[c - sxy];
    wm = A.wz[c - sxy];
  }
  for (int k = k0; k < k1; ++k, c += sxy) {
    const T wz = A.wz[c];  // 0 in the top layer
    const T yp = k < g.nz - 1 ? y[c + sxy] : T(0);
    T t = b[c] + (MODE == 2 ? A.gd[c] : A.g[c]) * yc;
    if (i > 0) t += A.wx[c - 1] * y[c - 1];
    if (i < nx - 1) t += A.wx[c] * y[c + 1];
    if (j > 0) t += A.wy[c - nx] * y[c - nx];
    if (j < g.ny - 1) t += A.wy[c] * y[c + nx];
    t += wm * ym;
    t += wz * yp;
    out[c] = MODE == 2 ? A.q[c] * t : t;
    ym = yc;
    wm = wz;
    yc = yp;
  }
}

// Launch shape of k_sc: lines as wide as the grid needs (up to 4 warps), and as many layers
// per thread (up to 4) as leave the SMs twice the threads they hold.
struct ScShape {
  dim3 grid;
  int threads, zc;
};
static ScShape sc_shape(const GridP& g) {
  ScShape s;
  s.threads = std::min(kLineThreads, (g.nx + 31) / 32 * 32);
  s.zc = 1;
  while (s.zc < 4 && g.n / (2 * s.zc) >= 2LL * kNumSM * 2048) s.zc *= 2;
  s.grid = dim3((unsigned)(g.ny * ((g.nz + s.zc - 1) / s.zc)), (unsigned)((g.nx + s.threads - 1) / s.threads), 1);
  return s;
}

// b = s r on the way in, z = s y on the way out, and without a pre-sweep r = q b.
template <class T>
__global__ void k_sc_in(long long n, const T* __restrict__ s, const double* __restrict__ r, T* __restrict__ b) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    b[i] = s[i] * (T)r[i];
}
template <class T>
__global__ void k_sc_out(long long n, const T* __restrict__ s, const T* __restrict__ y, double* __restrict__ z) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    z[i] = (double)(s[i] * y[i]);
}
template <class T>
__global__ void k_sc_mul(long long n, const T* __restrict__ q, const T* __restrict__ b, T* __restrict__ r) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    r[i] = q[i] * b[i];
}

// Hybrid Gauss-Seidel (the paper's smoother, Sec. 5.2 / Sec. 6): Gauss-Seidel inside
// the block one thread (or lane group) owns, Jacobi between blocks, scaled by
// a_ii + sum over couplings to other blocks of |a_ij| (the l1 form).  x == nullptr
// sweeps from zero; xo receives the new values (blocks read only x for each other).
//
// Finest level: a block is a segment of `seg` cells of one vertical column; the
// thread walks it upward (FWD) or downward carrying the new value of the cell just
// updated, so the in-block coupling costs no extra load.  Launch: blockIdx.x over
// (j, segment), blockIdx.y over x tiles, threadIdx.x = i (coalesced in x).
template <class T, bool FWD>
__global__ void __launch_bounds__(kLineThreads) k_hgs_st(GridP g, Stencil4<T> A, int seg, const T* __restrict__ b,
                                                         const T* __restrict__ x, T* __restrict__ xo) {
  int i = blockIdx.y * kLineThreads + threadIdx.x;
  if (i >= g.nx) return;
  int r = blockIdx.x;
  int j = r % g.ny;
  int k0 = (r / g.ny) * seg;
  int k1 = min(g.nz, k0 + seg);
  int nx = g.nx;
  int sxy = g.nx * g.ny;
  T carry = T(0);
  for (int q = 0; q < k1 - k0; ++q) {
    int k = FWD ? k0 + q : k1 - 1 - q;
    int c = (k * g.ny + j) * nx + i;
    T xc = x ? x[c] : T(0);
    T ax = A.diag[c] * xc;
    T d = A.diag[c];
    T w;
    if (i > 0) { w = A.wx[c - 1]; ax -= w * (x ? x[c - 1] : T(0)); d += w; }
    if (i < nx - 1) { w = A.wx[c]; ax -= w * (x ? x[c + 1] : T(0)); d += w; }
    if (j > 0) { w = A.wy[c - nx]; ax -= w * (x ? x[c - nx] : T(0)); d += w; }
    if (j < g.ny - 1) { w = A.wy[c]; ax -= w * (x ? x[c + nx] : T(0)); d += w; }
    if (k > 0) {
      w = A.wz[c - sxy];
      if (k - 1 >= k0) ax -= w * (FWD ? carry : (x ? x[c - sxy] : T(0)));  // in block: new below (FWD)
      else { ax -= w * (x ? x[c - sxy] : T(0)); d += w; }
    }
    if (k < g.nz - 1) {
      w = A.wz[c];
      if (k + 1 < k1) ax -= w * (FWD ? (x ? x[c + sxy] : T(0)) : carry);  // in block: new above (backward)
      else { ax -= w * (x ? x[c + sxy] : T(0)); d += w; }
    }
    T xn = xc + (b[c] - ax) / d;
    xo[c] = xn;
    carry = xn;
  }
}

// Coarser levels: a block is `bs` consecutive rows, walked by one group of G lanes
// (rows of tens to hundreds of entries); lane 0 writes each new value and the group
// synchronises before the next row reads it.
template <class T, bool FWD, int G>
__global__ void k_hgs_csr(int n, const int* __restrict__ rp, const int* __restrict__ col, const T* __restrict__ val,
                          int bs, const T* __restrict__ b, const T* __restrict__ x, T* __restrict__ xo) {
  int lane = threadIdx.x & (G - 1);
  unsigned mask = G == 32 ? 0xffffffffu : (((1u << G) - 1) << ((threadIdx.x & 31) & ~(G - 1)));
  int nblk = (n + bs - 1) / bs;
  int groups = (gridDim.x * blockDim.x) / G;
  for (int blk = (blockIdx.x * blockDim.x + threadIdx.x) / G; blk < nblk; blk += groups) {
    int r0 = blk * bs;
    int r1 = min(n, r0 + bs);
    for (int q = 0; q < r1 - r0; ++q) {
      int i = FWD ? r0 + q : r1 - 1 - q;
      T s = 0, d = 0;
      for (int e = rp[i] + lane; e < rp[i + 1]; e += G) {
        int jj = col[e];
        T a = val[e];
        T xv;
        if (jj >= r0 && jj < r1) {
          bool updated = FWD ? jj < i : jj > i;
          xv = updated ? xo[jj] : (x ? x[jj] : T(0));
          if (jj == i) d += a;
        } else {
          xv = x ? x[jj] : T(0);
          d += a < T(0) ? -a : a;
        }
        s += a * xv;
      }
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) {
        s += __shfl_down_sync(mask, s, o, G);
        d += __shfl_down_sync(mask, d, o, G);
      }
      if (lane == 0) xo[i] = (x ? x[i] : T(0)) + (b[i] - s) / d;
      __syncwarp(mask);
    }
  }
}

template <class T, bool FWD>
static void hgs_csr(cudaStream_t st, int n, long long nnz, const int* rp, const int* col, const T* val, int bs,
                    const T* b, const T* x, T* y) {
  double avg = n > 0 ? (double)nnz / n : 0.0;
  long long nblk = (n + bs - 1) / bs;
  if (avg > 64) k_hgs_csr<T, FWD, 32><<<grid_for(nblk * 32), kBlock, 0, st>>>(n, rp, col, val, bs, b, x, y);
  else if (avg > 24) k_hgs_csr<T, FWD, 16><<<grid_for(nblk * 16), kBlock, 0, st>>>(n, rp, col, val, bs, b, x, y);
  else if (avg > 10) k_hgs_csr<T, FWD, 8><<<grid_for(nblk * 8), kBlock, 0, st>>>(n, rp, col, val, bs, b, x, y);
  else k_hgs_csr<T, FWD, 4><<<grid_for(nblk * 4), kBlock, 0, st>>>(n, rp, col, val, bs, b, x, y);
}

template <class T>
static const Stencil4<T>& fine(rich_ctx* c);
template <>
const Stencil4<double>& fine<double>(rich_ctx* c) { return c->H.st64; }
template <>
const Stencil4<float>& fine<float>(rich_ctx* c) { return c->H.st32; }

template <class T>
static const ScaledSt<T>& scaled(rich_ctx* c);
template <>
const ScaledSt<double>& scaled<double>(rich_ctx* c) { return c->H.sc64; }
template <>
const ScaledSt<float>& scaled<float>(rich_ctx* c) { return c->H.sc32; }

template <class T>
struct LevelView {
  int n;
  const int *rp, *col;
  const T* val;
  const T* dinv;
  const int *prp, *pcol, *rrp, *rcol;
  const T *pval, *rval;
  SellSrc<T> sa, sp, sr;  // SELL sources of A, P, R
};

template <class T>
static LevelView<T> view(rich_ctx* c, int l);

template <>
LevelView<double> view<double>(rich_ctx* c, int l) {
  Level& L = c->H.lv[l];
  return LevelView<double>{L.n,     L.A.rowptr, L.A.col, L.A.val,
                           L.dinv,  L.P.rowptr, L.P.col, L.R.rowptr,
                           L.R.col, L.P.val,    L.R.val, {&L.sA, &L.A, L.A.val},
                           {&L.sP, &L.P, L.P.val}, {&L.sR, &L.R, L.R.val}};
}
template <>
LevelView<float> view<float>(rich_ctx* c, int l) {
  Level& L = c->H.lv[l];
  return LevelView<float>{L.n,       L.A.rowptr, L.A.col, L.A32,
                          L.dinv32,  L.P.rowptr, L.P.col, L.R.rowptr,
                          L.R.col,   L.P32,      L.R32,   {&L.sA, &L.A, L.A32},
                          {&L.sP, &L.P, L.P32},  {&L.sR, &L.R, L.R32}};
}

template <class T>
static const T* coarse_inv(rich_ctx* c);
template <>
const double* coarse_inv<double>(rich_ctx* c) { return c->H.cdense; }
template <>
const float* coarse_inv<float>(rich_ctx* c) { return c->H.cinv32; }

template <class T>
static int vcycle_level(rich_ctx* c, int l, const T* b, T** xres, bool first_done = false);

// One hybrid Gauss-Seidel sweep on level l (x == nullptr: from zero) into xo.
template <class T>
static int hgs_sweep(rich_ctx* c, int l, bool forward, const T* b, const T* x, T* xo) {
  Hierarchy& H = c->H;
  Level& L = H.lv[l];
  const double es = sizeof(T);
  if (l == 0) {
    const GridP& g = c->g;
    int nseg = (g.nz + H.opts.hgs_seg - 1) / H.opts.hgs_seg;
    dim3 grid((unsigned)((long long)g.ny * nseg), (unsigned)((g.nx + kLineThreads - 1) / kLineThreads), 1);
    ProfScope ps("hgs_l0", c->st, (double)g.n * (x ? 8.0 : 7.0) * es, 20.0 * (double)g.n);
    if (forward) k_hgs_st<T, true><<<grid, kLineThreads, 0, c->st>>>(g, fine<T>(c), H.opts.hgs_seg, b, x, xo);
    else k_hgs_st<T, false><<<grid, kLineThreads, 0, c->st>>>(g, fine<T>(c), H.opts.hgs_seg, b, x, xo);
  } else {
    LevelView<T> v = view<T>(c, l);
    ProfScope ps("hgs", c->st, (double)L.n * (4.0 + 3.0 * es) + (double)L.A.nnz * (4.0 + es), 4.0 * L.A.nnz);
    if (forward) hgs_csr<T, true>(c->st, L.n, L.A.nnz, v.rp, v.col, v.val, H.opts.hgs_block, b, x, xo);
    else hgs_csr<T, false>(c->st, L.n, L.A.nnz, v.rp, v.col, v.val, H.opts.hgs_block, b, x, xo);
  }
  RICH_LAUNCH_CHECK();
  return RICH_OK;
}

// V-cycle level with hybrid Gauss-Seidel: nu1 backward sweeps (the first from zero),
// residual, restriction, coarse correction, nu2 forward sweeps.
template <class T>
static int vcycle_level_hgs(rich_ctx* c, int l, const T* b, T** xres) {
  Hierarchy& H = c->H;
  Level& L = H.lv[l];
  LevelView<T> v = view<T>(c, l);
  int n = v.n;
  int g = grid_for(n);
  T* x = (T*)L.x;
  T* t = (T*)L.t;
  const double es = sizeof(T);
  const bool st0 = (l == 0);
  for (int s = 0; s < H.opts.nu1; ++s) {
    RICH_CHECK(hgs_sweep<T>(c, l, false, b, s == 0 ? (const T*)nullptr : (const T*)x, t));
    std::swap(x, t);
  }
  if (H.opts.nu1 == 0) RICH_CUDA(cudaMemsetAsync(x, 0, sizeof(T) * n, c->st));
  {
    ProfScope ps(st0 ? "resid_l0" : "csr_resid", c->st,
                 st0 ? (double)n * 7.0 * es : (double)n * (4.0 + 3.0 * es) + (double)L.A.nnz * (4.0 + es));
    if (st0) k_st_resid<T><<<line_grid(c->g), kLineThreads, 0, c->st>>>(c->g, fine<T>(c), b, x, (T*)L.r);
    else RICH_CHECK(csr_op<T, 3>(c, n, L.A.nnz, v.rp, v.col, v.val, (const T*)nullptr, b, x, (T*)L.r, &v.sa));
  }
  RICH_LAUNCH_CHECK();
  Level& C = H.lv[l + 1];
  {
    ProfScope ps("restrict", c->st, (double)C.n * (4.0 + es) + (double)L.R.nnz * (4.0 + es) + (double)n * es);
    RICH_CHECK(csr_op<T, 0>(c, C.n, L.R.nnz, v.rrp, v.rcol, v.rval, (const T*)nullptr, (const T*)nullptr,
                            (const T*)L.r, (T*)C.b, &v.sr));
  }
  RICH_LAUNCH_CHECK();
  T* xc = nullptr;
  RICH_CHECK(vcycle_level<T>(c, l + 1, (const T*)C.b, &xc));
  {
    ProfScope ps("prolong", c->st, (double)n * (4.0 + 2.0 * es) + (double)L.P.nnz * (4.0 + es) + (double)C.n * es);
    RICH_CHECK(csr_op<T, 1>(c, n, L.P.nnz, v.prp, v.pcol, v.pval, (const T*)nullptr, (const T*)nullptr, xc, x,
                            &v.sp));
  }
  RICH_LAUNCH_CHECK();
  for (int s = 0; s < H.opts.nu2; ++s) {
    RICH_CHECK(hgs_sweep<T>(c, l, true, b, x, t));
    std::swap(x, t);
  }
  if (x != (T*)L.x) {
    L.t = L.x;
    L.x = x;
  }
  *xres = x;
  return RICH_OK;
}

// b is the level's right-hand side, the result is left in *xres (one of the level's buffers).
// first_done: the level's x holds the first sweep, D_l1^-1 b, already (the restriction's y2;
// with nu1 > 0 on every level below the finest but a dense coarsest one).
template <class T>
static int vcycle_level(rich_ctx* c, int l, const T* b, T** xres, bool first_done) {
  Hierarchy& H = c->H;
  Level& L = H.lv[l];
  LevelView<T> v = view<T>(c, l);
  int n = v.n;
  int g = grid_for(n);
  T* x = (T*)L.x;
  T* t = (T*)L.t;
  const double es = sizeof(T);
  // algorithmic bytes of one sweep over this level's CSR matrix (pattern + values + 4 vectors)
  const double sweep_bytes = (double)n * (4.0 + 4.0 * es) + (double)L.A.nnz * (4.0 + es);
  if (l == H.nlev - 1) {
    if (H.dense) {
      ProfScope ps("coarse_gemv", c->st, (double)n * n * es + 2.0 * n * es);
      k_gemv<T><<<grid_for((long long)n * 32), kBlock, 0, c->st>>>(n, coarse_inv<T>(c), b, x);
      RICH_LAUNCH_CHECK();
    } else {  // stalled coarsening: l1-Jacobi sweeps from zero on the (large) coarsest level
      if (!first_done) {
        k_jacobi0<T><<<g, kBlock, 0, c->st>>>(n, v.dinv, b, x);
        RICH_LAUNCH_CHECK();
      }
      for (int s = 1; s < kCoarseSweeps; ++s) {
        RICH_CHECK(csr_op<T, 2>(c, n, L.A.nnz, v.rp, v.col, v.val, v.dinv, b, x, t, &v.sa));
        RICH_LAUNCH_CHECK();
        std::swap(x, t);
      }
    }
    *xres = x;
    return RICH_OK;
  }
  int nu1 = H.opts.nu1, nu2 = H.opts.nu2;
  if (H.opts.smoother == RICH_SMOOTH_HYBRID_GS) return vcycle_level_hgs<T>(c, l, b, xres);
  // the finest level in scaled form (H.scaled holds here: l1-Jacobi, more than one level)
  const bool st0 = (l == 0);
  const ScaledSt<T>& S = scaled<T>(c);
  const ScShape sh = sc_shape(c->g);
  const double st_bytes = (double)n * 7.0 * es;  // g, 3 face weights, b, y in; y out
  auto sweep = [&](const T* from, T* to) -> int {
    {
      ProfScope ps(st0 ? "l1jacobi_l0" : "l1jacobi", c->st, st0 ? st_bytes : sweep_bytes,
                   st0 ? 14.0 * n : 2.0 * L.A.nnz + 3.0 * n);
      if (st0) k_sc<T, 1><<<sh.grid, sh.threads, 0, c->st>>>(c->g, S, sh.zc, b, from, to);
      else RICH_CHECK(csr_op<T, 2>(c, n, L.A.nnz, v.rp, v.col, v.val, v.dinv, b, from, to, &v.sa));
    }
    RICH_LAUNCH_CHECK();
    return RICH_OK;
  };
  // where the iterate is: the first sweep from x = 0 gives b itself on the finest level, and
  // below it x holds it already (first_done)
  const T* cur = x;
  if (nu1 > 0) {
    if (st0) cur = b;
    for (int s = 1; s < nu1; ++s) {
      T* to = cur == x ? t : x;
      RICH_CHECK(sweep(cur, to));
      if (to == t) std::swap(x, t);
      cur = x;
    }
    {
      ProfScope ps(st0 ? "resid_l0" : "csr_resid", c->st,
                   st0 ? st_bytes + (double)n * es : sweep_bytes - (double)n * es,
                   st0 ? 16.0 * n : 0.0);
      if (st0) k_sc<T, 2><<<sh.grid, sh.threads, 0, c->st>>>(c->g, S, sh.zc, b, cur, (T*)L.r);
      else RICH_CHECK(csr_op<T, 3>(c, n, L.A.nnz, v.rp, v.col, v.val, (const T*)nullptr, b, cur, (T*)L.r, &v.sa));
    }
    RICH_LAUNCH_CHECK();
  } else {
    RICH_CUDA(cudaMemsetAsync(x, 0, sizeof(T) * n, c->st));
    if (st0) {
      k_sc_mul<T><<<g, kBlock, 0, c->st>>>(n, S.q, b, (T*)L.r);
      RICH_LAUNCH_CHECK();
    } else {
      RICH_CUDA(cudaMemcpyAsync(L.r, b, sizeof(T) * n, cudaMemcpyDeviceToDevice, c->st));
    }
  }
  // the next level's first sweep rides on the restriction: one launch less per level and
  // cycle (48^3 MIXED FCG: 1935 -> 1892 us, eight 32^3 soils: 20.3 -> 19.8 ms)
  const bool first_next = nu1 > 0 && !(l + 2 == H.nlev && H.dense);
  Level& C = H.lv[l + 1];
  {
    ProfScope ps("restrict", c->st, (double)C.n * (4.0 + es) + (double)L.R.nnz * (4.0 + es) + (double)n * es);
    RICH_CHECK(csr_op<T, 0>(c, C.n, L.R.nnz, v.rrp, v.rcol, v.rval, view<T>(c, l + 1).dinv, (const T*)nullptr,
                            (const T*)L.r, (T*)C.b, &v.sr, first_next ? (T*)C.x : (T*)nullptr));
  }
  RICH_LAUNCH_CHECK();
  T* xc = nullptr;
  RICH_CHECK(vcycle_level<T>(c, l + 1, (const T*)C.b, &xc, first_next));
  {
    ProfScope ps("prolong", c->st, (double)n * (4.0 + 2.0 * es) + (double)L.P.nnz * (4.0 + es) + (double)C.n * es);
    if (st0)  // y = cur + q (P xc)
      RICH_CHECK(csr_op<T, 4>(c, n, L.P.nnz, v.prp, v.pcol, v.pval, S.q, cur, xc, x, &v.sp));
    else
      RICH_CHECK(csr_op<T, 1>(c, n, L.P.nnz, v.prp, v.pcol, v.pval, (const T*)nullptr, (const T*)nullptr, xc, x,
                              &v.sp));
  }
  RICH_LAUNCH_CHECK();
  for (int s = 0; s < nu2; ++s) {
    RICH_CHECK(sweep(x, t));
    std::swap(x, t);
  }
  // keep the level's buffer pointers consistent with where the result lives
  if (x != (T*)L.x) {
    L.t = L.x;
    L.x = x;
  }
  *xres = x;
  return RICH_OK;
}

// Captures the V-cycle from the level-0 right-hand side buffer L0.b as one graph
// (H.vc_exec, its result at H.vc_out).  It runs after a direct application, so the
// tuner's choices and the SELL copies exist and nothing in the cycle allocates or
// synchronises.  The capture stream is a private non-blocking one (the context's
// stream may be the legacy default stream, which cannot be captured).  A failed
// capture leaves direct launches for the rest of this hierarchy.
static int vcycle_capture(rich_ctx* c) {
  Hierarchy& H = c->H;
  Level& L0 = H.lv[0];
  cudaStream_t cs;
  RICH_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
  cudaStream_t saved = c->st;
  RICH_CUDA(cudaStreamSynchronize(saved));
  c->st = cs;
  long long before = 0, after = 0;
  rich_kernel_launches(&before);
  cudaGraph_t graph = nullptr;
  void* out = nullptr;
  int rc = RICH_OK;
  cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    if (c->prec == RICH_PREC_MIXED) {
      float* x = nullptr;
      rc = vcycle_level<float>(c, 0, (const float*)L0.b, &x);
      out = x;
    } else {
      double* x = nullptr;
      rc = vcycle_level<double>(c, 0, (const double*)L0.b, &x);
      out = x;
    }
    e = cudaStreamEndCapture(cs, &graph);
  }
  c->st = saved;
  rich_kernel_launches(&after);
  count_launches(before - after);  // recorded, not launched
  if (e == cudaSuccess && rc == RICH_OK) {
    e = cudaGraphInstantiate(&H.vc_exec, graph, 0);
    if (e == cudaSuccess) {
      H.vc_nodes = after - before;
      H.vc_out = out;
    } else {
      H.vc_exec = nullptr;
    }
  }
  if (graph) cudaGraphDestroy(graph);
  cudaStreamDestroy(cs);
  if (e != cudaSuccess || rc != RICH_OK || !H.vc_exec) {
    cudaGetLastError();
    if (H.vc_exec) cudaGraphExecDestroy(H.vc_exec);
    H.vc_exec = nullptr;
    H.vc_off = true;
  }
  return RICH_OK;
}

// The level-0 right-hand side from r, and the result x into z.
static int vcycle_in(rich_ctx* c, const double* r) {
  const Hierarchy& H = c->H;
  const Level& L0 = H.lv[0];
  const long long n = c->g.n;
  const int g = grid_for(n);
  if (H.scaled) {
    if (c->prec == RICH_PREC_MIXED) k_sc_in<float><<<g, kBlock, 0, c->st>>>(n, H.sc32.s, r, (float*)L0.b);
    else k_sc_in<double><<<g, kBlock, 0, c->st>>>(n, H.sc64.s, r, (double*)L0.b);
    RICH_LAUNCH_CHECK();
  } else if (c->prec == RICH_PREC_MIXED) {
    k_d2f<<<g, kBlock, 0, c->st>>>(n, r, (float*)L0.b);
    RICH_LAUNCH_CHECK();
  } else {
    RICH_CUDA(cudaMemcpyAsync(L0.b, r, sizeof(double) * n, cudaMemcpyDeviceToDevice, c->st));
  }
  return RICH_OK;
}
static int vcycle_out(rich_ctx* c, const void* x, double* z) {
  const Hierarchy& H = c->H;
  const long long n = c->g.n;
  const int g = grid_for(n);
  if (H.scaled) {
    if (c->prec == RICH_PREC_MIXED) k_sc_out<float><<<g, kBlock, 0, c->st>>>(n, H.sc32.s, (const float*)x, z);
    else k_sc_out<double><<<g, kBlock, 0, c->st>>>(n, H.sc64.s, (const double*)x, z);
    RICH_LAUNCH_CHECK();
  } else if (c->prec == RICH_PREC_MIXED) {
    k_f2d<<<g, kBlock, 0, c->st>>>(n, (const float*)x, z);
    RICH_LAUNCH_CHECK();
  } else {
    RICH_CUDA(cudaMemcpyAsync(z, x, sizeof(double) * n, cudaMemcpyDeviceToDevice, c->st));
  }
  return RICH_OK;
}

// The V-cycle's kernels from the level-0 right-hand side into z, launched (or captured) as
// they come.
static int vcycle_direct(rich_ctx* c, double* z) {
  Level& L0 = c->H.lv[0];
  if (c->prec == RICH_PREC_MIXED) {
    float* x = nullptr;
    RICH_CHECK(vcycle_level<float>(c, 0, (const float*)L0.b, &x));
    return vcycle_out(c, x, z);
  }
  double* x = nullptr;
  RICH_CHECK(vcycle_level<double>(c, 0, (const double*)L0.b, &x));
  return vcycle_out(c, x, z);
}

// Whether the V-cycle of this hierarchy may run from a captured graph now.
static bool vcycle_graphable(rich_ctx* c) {
  const Hierarchy& H = c->H;
  return H.opts.graph && H.opts.precond == RICH_PRECOND_AMG && H.opts.smoother == RICH_SMOOTH_L1JACOBI && !H.vc_off &&
         !profiling_active();
}

// The V-cycle on the staged right-hand side (the level-0 buffer b) into z.
static int vcycle_staged(rich_ctx* c, double* z) {
  Hierarchy& H = c->H;
  if (vcycle_graphable(c) && H.vc_calls > 0) {  // the first application launched directly
    if (!H.vc_exec) RICH_CHECK(vcycle_capture(c));
    if (H.vc_exec) {
      RICH_CUDA(cudaGraphLaunch(H.vc_exec, c->st));
      count_launches(H.vc_nodes);
      return vcycle_out(c, H.vc_out, z);
    }
  }
  ++H.vc_calls;
  return vcycle_direct(c, z);
}

int vcycle_apply(rich_ctx* c, const double* r, double* z) {
  if (!c->H.built) return RICH_ESTATE;
  if (c->H.opts.precond == RICH_PRECOND_AS) return as_apply(c, r, z);
  RICH_CHECK(vcycle_in(c, r));
  return vcycle_staged(c, z);
}

// ---------------------------------------------------------------- Krylov kernels (FP64)

// y += sign * sum_q coef[q] V[q]
__global__ void k_multiaxpy(long long n, int nv, const double* __restrict__ V, const double* __restrict__ coef,
                            double sign, double* __restrict__ y) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int q = 0; q < nv; ++q) s += coef[q] * V[(long long)q * n + i];
    y[i] += sign * s;
  }
}

__global__ void k_scale(long long n, const double* __restrict__ a, double f, double* __restrict__ b) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    b[i] = f * a[i];
}

// y = a - b
__global__ void k_sub(long long n, const double* __restrict__ a, const double* __restrict__ b, double* __restrict__ y) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = a[i] - b[i];
}

// y = a + lam * d
__global__ void k_axpby(long long n, const double* __restrict__ a, double lam, const double* __restrict__ d,
                        double* __restrict__ y) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = a[i] + lam * d[i];
}

static int ensure_krylov(rich_ctx* c, int m) {
  KrylovWork& k = c->kw;
  long long n = c->g.n;
  if (k.n != n) {
    dfree(k.x); dfree(k.r); dfree(k.p); dfree(k.q); dfree(k.z); dfree(k.w);
    RICH_CHECK(dalloc(&k.x, n));
    RICH_CHECK(dalloc(&k.r, n));
    RICH_CHECK(dalloc(&k.p, n));
    RICH_CHECK(dalloc(&k.q, n));
    RICH_CHECK(dalloc(&k.z, n));
    RICH_CHECK(dalloc(&k.w, n));
    RICH_CHECK(dalloc(&k.hcoef, 128));
    k.n = n;
  }
  if (m > 0 && !k.gram) RICH_CHECK(dalloc(&k.gram, kGsLd * kGsLd));
  if (m > 0 && !k.peak) RICH_CHECK(dalloc(&k.peak, kGsLd));
  if (m > 0 && k.m < m) {
    dfree(k.V);
    dfree(k.Z);
    RICH_CHECK(dalloc(&k.V, (long long)(m + 1) * n));
    RICH_CHECK(dalloc(&k.Z, (long long)m * n));
    k.m = m;
  }
  return RICH_OK;
}

// ---------------------------------------------------------------- flexible CG on the device
// Notay's flexible CG (truncation 1), for one problem or S of them stacked along z, each
// with its own scalars, tests and iteration count; a problem that has stopped is frozen.
// An iteration is the V-cycle and four kernels: z and z . q_prev, the direction, q = J p
// with p . q and p . r, and the update with ||r||^2, whose last block makes the decisions
// (convergence, (p, q) <= 0, growth, stagnation, maxit) and writes the next right-hand
// side's scaling in the same pass.  The iterations are the body of a WHILE node of a CUDA
// graph, which the last block continues or ends: no host turn-round (about 10 us) and no
// launches (0.75 us per kernel) between iterations, 2.5 us for the loop.
// 48^3 MIXED, V(1,1): 27 launches and a synchronisation took 78 us per iteration.
struct FcgSeg {
  double zq, pq, pr, pq_prev;            // of the iteration under way; (p, q) of the last one
  double rn, bn, target, best, window;   // ||r||, ||b||, the tests' references
  int it, reason;                        // iterations; why it stopped (kFcg...), 0 while running
};
struct FcgOut {  // pinned mirror
  double rn, bn;
  int it, reason;
};
constexpr int kFcgMaxSeg = 32;
struct FcgDev {
  FcgSeg seg[kFcgMaxSeg];
  double stall;
  int maxit;
};
// 1..4 are KrylovWork::fail_reason's
constexpr int kFcgConverged = 10, kFcgZero = 11, kFcgNonfinite = 12;
constexpr int kFcgThreads = 256;
static_assert(sizeof(FcgOut) * kFcgMaxSeg <= kPinnedBlock, "the mirror is one pinned block");

// Blocks per problem: two per SM in all, fewer where there are fewer cells.
static int fcg_blocks(long long ns, int S) {
  const long long most = std::max(1, 2 * kNumSM / S);
  return (int)std::min(most, (ns + kFcgThreads - 1) / kFcgThreads);
}

// Block sums v of this block's problem to the partials; in the last block to finish, the
// totals of every problem, tot[q * S + s], in block order.
template <int NQ>
__device__ __forceinline__ bool fcg_sums(double (&v)[NQ], double* part, unsigned* ticket, double* tot) {
  constexpr int W = kFcgThreads / 32;
  __shared__ double sh[W][NQ];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nb = gridDim.x, S = gridDim.y;
#pragma unroll
  for (int q = 0; q < NQ; ++q)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
  if (lane == 0)
    for (int q = 0; q < NQ; ++q) sh[wid][q] = v[q];
  __syncthreads();
  if (threadIdx.x < NQ) {
    double t = 0.0;
    for (int w = 0; w < W; ++w) t += sh[w][threadIdx.x];
    part[((long long)threadIdx.x * S + blockIdx.y) * nb + blockIdx.x] = t;
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == (unsigned)(nb * S) - 1;
  __syncthreads();
  if (!last) return false;
  __threadfence();
  for (int i = wid; i < NQ * S; i += W) {
    double t = 0.0;
    for (int k = lane; k < nb; k += 32) t += __ldcg(&part[(long long)i * nb + k]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) tot[i] = t;
  }
  if (threadIdx.x == 0) *ticket = 0;
  __syncthreads();
  return true;
}

// x = 0, r = b, the V-cycle's right-hand side; ||b|| and the tests' references.
template <class T>
__global__ void __launch_bounds__(kFcgThreads) k_fcg_begin(long long ns, const double* __restrict__ b,
                                                           double* __restrict__ x, double* __restrict__ r,
                                                           const T* __restrict__ sc, T* __restrict__ vb, double eta,
                                                           double stall, int maxit, FcgDev* __restrict__ dev,
                                                           double* __restrict__ part, unsigned* __restrict__ ticket,
                                                           FcgOut* __restrict__ out) {
  __shared__ double tot[kFcgMaxSeg];
  const long long base = blockIdx.y * ns;
  double v[1] = {0.0};
  for (long long i = blockIdx.x * (long long)kFcgThreads + threadIdx.x; i < ns;
       i += (long long)gridDim.x * kFcgThreads) {
    const double t = b[base + i];
    x[base + i] = 0.0;
    r[base + i] = t;
    if (vb) vb[base + i] = sc[base + i] * (T)t;
    v[0] = fma(t, t, v[0]);
  }
  if (!fcg_sums<1>(v, part, ticket, tot)) return;
  if (threadIdx.x == 0) {
    dev->stall = stall;
    dev->maxit = maxit;
  }
  if (threadIdx.x < gridDim.y) {
    FcgSeg s{};
    s.bn = s.rn = s.best = s.window = sqrt(tot[threadIdx.x]);
    s.target = eta * s.bn;
    if (!isfinite(s.bn)) s.reason = kFcgNonfinite;
    else if (!(s.bn > 0)) s.reason = kFcgZero;
    else if (maxit < 1) s.reason = 1;  // a batch's limit of no iterations at all: x = 0, not converged
    dev->seg[threadIdx.x] = s;
    out[threadIdx.x] = FcgOut{s.rn, s.bn, 0, s.reason};
  }
}

// z = sc y (given y; else z is there already) and z . q_prev.
template <class T>
__global__ void __launch_bounds__(kFcgThreads) k_fcg_z(long long ns, const T* __restrict__ sc, const T* __restrict__ y,
                                                       double* __restrict__ z, const double* __restrict__ q,
                                                       FcgDev* __restrict__ dev, double* __restrict__ part,
                                                       unsigned* __restrict__ ticket) {
  __shared__ double tot[kFcgMaxSeg];
  const long long base = blockIdx.y * ns;
  const bool first = dev->seg[blockIdx.y].it == 0;  // no q yet
  double v[1] = {0.0};
  for (long long i = base + blockIdx.x * (long long)kFcgThreads + threadIdx.x; i < base + ns;
       i += (long long)gridDim.x * kFcgThreads) {
    double t;
    if (y) {
      t = (double)(sc[i] * y[i]);
      z[i] = t;
    } else {
      t = z[i];
    }
    if (!first) v[0] = fma(t, q[i], v[0]);
  }
  if (fcg_sums<1>(v, part, ticket, tot) && threadIdx.x < gridDim.y) dev->seg[threadIdx.x].zq = tot[threadIdx.x];
}

// p = z - (zq / pq_prev) p; the first direction is z.
__global__ void k_fcg_dir(long long ns, const double* __restrict__ z, double* __restrict__ p,
                          const FcgDev* __restrict__ dev) {
  const FcgSeg& s = dev->seg[blockIdx.y];
  if (s.reason) return;
  const bool first = s.it == 0;
  const double beta = first ? 0.0 : s.zq / s.pq_prev;
  const long long base = blockIdx.y * ns;
  for (long long i = base + blockIdx.x * (long long)blockDim.x + threadIdx.x; i < base + ns;
       i += (long long)gridDim.x * blockDim.x)
    p[i] = first ? z[i] : z[i] - beta * p[i];
}

// q = J p, p . q and p . r.
__global__ void __launch_bounds__(kFcgThreads) k_fcg_apply(GridP g, long long ns, const double* __restrict__ J,
                                                           const double* __restrict__ p, const double* __restrict__ r,
                                                           double* __restrict__ q, FcgDev* __restrict__ dev,
                                                           double* __restrict__ part, unsigned* __restrict__ ticket) {
  __shared__ double tot[2 * kFcgMaxSeg];
  const long long n = g.n;
  const int sxy = g.nx * g.ny, base = (int)(blockIdx.y * ns);
  double v[2] = {0.0, 0.0};
  for (int l = blockIdx.x * kFcgThreads + threadIdx.x; l < (int)ns; l += gridDim.x * kFcgThreads) {
    const int c = base + l, row = c / g.nx, i = c - row * g.nx, k = row / g.ny, j = row - k * g.ny, kl = k % g.nzs;
    const double pc = p[c];
    double t = J[c] * pc;
    if (i > 0) t += J[n + c] * p[c - 1];
    if (i < g.nx - 1) t += J[2 * n + c] * p[c + 1];
    if (j > 0) t += J[3 * n + c] * p[c - g.nx];
    if (j < g.ny - 1) t += J[4 * n + c] * p[c + g.nx];
    if (kl > 0) t += J[5 * n + c] * p[c - sxy];
    if (kl < g.nzs - 1) t += J[6 * n + c] * p[c + sxy];
    q[c] = t;
    v[0] = fma(pc, t, v[0]);
    v[1] = fma(pc, r[c], v[1]);
  }
  if (fcg_sums<2>(v, part, ticket, tot) && threadIdx.x < gridDim.y) {
    dev->seg[threadIdx.x].pq = tot[threadIdx.x];
    dev->seg[threadIdx.x].pr = tot[gridDim.y + threadIdx.x];
  }
}

// x += alpha p, r -= alpha q, the V-cycle's next right-hand side; then the tests.
template <class T>
__global__ void __launch_bounds__(kFcgThreads) k_fcg_update(long long ns, double* __restrict__ x,
                                                            double* __restrict__ r, const double* __restrict__ p,
                                                            const double* __restrict__ q, const T* __restrict__ sc,
                                                            T* __restrict__ vb, FcgDev* __restrict__ dev,
                                                            double* __restrict__ part, unsigned* __restrict__ ticket,
                                                            FcgOut* __restrict__ out,
                                                            cudaGraphConditionalHandle loop, int looped) {
  __shared__ double tot[kFcgMaxSeg];
  __shared__ int running, bad;
  const long long base = blockIdx.y * ns;
  double v[1] = {0.0};
  if (dev->seg[blockIdx.y].reason == 0) {
    const double alpha = dev->seg[blockIdx.y].pr / dev->seg[blockIdx.y].pq;
    for (long long i = base + blockIdx.x * (long long)kFcgThreads + threadIdx.x; i < base + ns;
         i += (long long)gridDim.x * kFcgThreads) {
      x[i] += alpha * p[i];
      const double t = r[i] - alpha * q[i];
      r[i] = t;
      if (vb) vb[i] = sc[i] * (T)t;
      v[0] = fma(t, t, v[0]);
    }
  }
  if (threadIdx.x == 0) running = bad = 0;
  if (!fcg_sums<1>(v, part, ticket, tot)) return;
  if (threadIdx.x < gridDim.y) {
    FcgSeg& s = dev->seg[threadIdx.x];
    if (s.reason == 0) {
      const double rn = sqrt(tot[threadIdx.x]);
      ++s.it;
      s.rn = rn;
      s.pq_prev = s.pq;
      if (!isfinite(rn) || !isfinite(s.pq)) s.reason = kFcgNonfinite;
      else if (!(s.pq > 0)) s.reason = 2;
      else if (rn <= s.target) s.reason = kFcgConverged;
      else if (rn > 10.0 * s.best) s.reason = 3;
      else if (s.it % kStallWindow == 0) {  // stagnation over the last window
        if (dev->stall > 0 && rn > (1.0 - dev->stall) * s.window) s.reason = 4;
        s.window = rn;
      }
      if (s.reason == 0 && s.it >= dev->maxit) s.reason = 1;
      s.best = fmin(s.best, rn);
      out[threadIdx.x] = FcgOut{rn, s.bn, s.it, s.reason};
    }
    if (s.reason == 0) atomicOr(&running, 1);
    if (s.reason == kFcgNonfinite) atomicOr(&bad, 1);
  }
  __syncthreads();
  if (threadIdx.x == 0 && looped) cudaGraphSetConditional(loop, running && !bad ? 1 : 0);
}

template <class T>
static T* vcycle_rhs(rich_ctx* c) { return c->H.scaled ? (T*)c->H.lv[0].b : nullptr; }

// One iteration on S problems, launched or captured as it comes.
template <class T>
static int fcg_body(rich_ctx* c, int S, cudaGraphConditionalHandle loop, int looped) {
  KrylovWork& k = c->kw;
  Hierarchy& H = c->H;
  const long long n = c->g.n, ns = n / S;
  const dim3 grid(fcg_blocks(ns, S), S);
  const T* sc = scaled<T>(c).s;
  FcgDev* dev = static_cast<FcgDev*>(k.fcg);
  FcgOut* out = static_cast<FcgOut*>(k.fcg_out);
  const T* y = nullptr;
  if (H.opts.precond == RICH_PRECOND_AS) {
    RICH_CHECK(as_apply(c, k.r, k.z));
  } else {
    if (!H.scaled) RICH_CHECK(vcycle_in(c, k.r));
    T* res = nullptr;
    RICH_CHECK(vcycle_level<T>(c, 0, (const T*)H.lv[0].b, &res));
    if (H.scaled) y = res;
    else RICH_CHECK(vcycle_out(c, res, k.z));
  }
  k_fcg_z<T><<<grid, kFcgThreads, 0, c->st>>>(ns, sc, y, k.z, k.q, dev, c->partials, c->ticket);
  RICH_LAUNCH_CHECK();
  k_fcg_dir<<<dim3(grid_for(ns), S), kBlock, 0, c->st>>>(ns, k.z, k.p, dev);
  RICH_LAUNCH_CHECK();
  {
    ProfScope ps("stencil_spmv", c->st, (double)n * 80.0, (double)n * 17.0);
    k_fcg_apply<<<grid, kFcgThreads, 0, c->st>>>(c->g, ns, c->J7, k.p, k.r, k.q, dev, c->partials, c->ticket);
  }
  RICH_LAUNCH_CHECK();
  {
    ProfScope ps("fcg_update", c->st, (double)n * 48.0);
    k_fcg_update<T><<<grid, kFcgThreads, 0, c->st>>>(ns, k.x, k.r, k.p, k.q, sc, vcycle_rhs<T>(c), dev, c->partials,
                                                     c->ticket, out, loop, looped);
  }
  RICH_LAUNCH_CHECK();
  return RICH_OK;
}

// Which of the hierarchy's loops serves S problems (S is 1 or the context's nbatch).
static int fcg_slot(int S) { return S > 1; }

// Captures the loop: a WHILE node whose body is fcg_body.  As for the V-cycle, on a private
// stream after a direct application; a failure leaves direct launches.
template <class T>
static void fcg_capture(rich_ctx* c, int S) {
  Hierarchy& H = c->H;
  cudaStream_t cs = nullptr;
  cudaGraph_t graph = nullptr, body = nullptr;
  cudaStream_t saved = c->st;
  long long before = 0, after = 0;
  int rc = RICH_OK;
  cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaStreamSynchronize(saved);
  if (e == cudaSuccess) e = cudaGraphCreate(&graph, 0);
  cudaGraphConditionalHandle loop;
  if (e == cudaSuccess) e = cudaGraphConditionalHandleCreate(&loop, graph, 1, cudaGraphCondAssignDefault);
  if (e == cudaSuccess) {
    cudaGraphNodeParams np = {};
    np.type = cudaGraphNodeTypeConditional;
    np.conditional.handle = loop;
    np.conditional.type = cudaGraphCondTypeWhile;
    np.conditional.size = 1;
    cudaGraphNode_t node;
    e = cudaGraphAddNode(&node, graph, nullptr, nullptr, 0, &np);
    if (e == cudaSuccess) body = np.conditional.phGraph_out[0];
  }
  if (e == cudaSuccess)
    e = cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    rich_kernel_launches(&before);
    c->st = cs;
    rc = fcg_body<T>(c, S, loop, 1);
    c->st = saved;
    rich_kernel_launches(&after);
    count_launches(before - after);  // recorded, not launched
    cudaGraph_t captured = nullptr;
    e = cudaStreamEndCapture(cs, &captured);  // the body itself
  }
  cudaGraphExec_t& exec = H.fcg_exec[fcg_slot(S)];
  if (e == cudaSuccess && rc == RICH_OK) {
    e = cudaGraphInstantiate(&exec, graph, 0);
    if (e == cudaSuccess) H.fcg_nodes[fcg_slot(S)] = after - before;
    else exec = nullptr;
  }
  if (graph) cudaGraphDestroy(graph);
  if (cs) cudaStreamDestroy(cs);
  if (e != cudaSuccess || rc != RICH_OK || !exec) {
    cudaGetLastError();
    exec = nullptr;
    H.fcg_off = true;
  }
}

template <class T>
static int fcg_solve(rich_ctx* c, int S, const double* b, double* x, const rich_krylov_opts* o) {
  KrylovWork& k = c->kw;
  Hierarchy& H = c->H;
  const long long n = c->g.n, ns = n / S;
  if (!k.fcg) {
    FcgDev* d = nullptr;
    RICH_CHECK(dalloc(&d, 1));
    k.fcg = d;
  }
  if (!k.fcg_out && !(k.fcg_out = pinned_get())) return RICH_ENOMEM;
  const FcgOut* out = static_cast<const FcgOut*>(k.fcg_out);
  k_fcg_begin<T><<<dim3(fcg_blocks(ns, S), S), kFcgThreads, 0, c->st>>>(
      ns, b, k.x, k.r, scaled<T>(c).s, vcycle_rhs<T>(c), o->eta, o->stall, o->maxit, static_cast<FcgDev*>(k.fcg),
      c->partials, c->ticket, static_cast<FcgOut*>(k.fcg_out));
  RICH_LAUNCH_CHECK();
  auto running = [&]() {
    bool any = false;
    for (int s = 0; s < S; ++s) {
      if (out[s].reason == kFcgNonfinite) return false;
      any = any || out[s].reason == 0;
    }
    return any;
  };
  const bool graphs = vcycle_graphable(c) && !H.fcg_off;
  bool waited = false;
  for (;;) {
    if (graphs && !H.fcg_off && H.vc_calls > 0) {  // a first application launched directly
      if (waited && !running()) break;
      if (!H.fcg_exec[fcg_slot(S)]) fcg_capture<T>(c, S);
      if (H.fcg_exec[fcg_slot(S)]) {
        auto most = [&]() {  // iterations of the problem that went longest
          int it = 0;
          for (int s = 0; s < S; ++s) it = std::max(it, out[s].it);
          return it;
        };
        const int it0 = waited ? most() : 0;
        RICH_CUDA(cudaGraphLaunch(H.fcg_exec[fcg_slot(S)], c->st));
        RICH_CUDA(cudaStreamSynchronize(c->st));
        count_launches(std::max(1, most() - it0) * H.fcg_nodes[fcg_slot(S)]);
        break;
      }
    }
    if (!waited) RICH_CUDA(cudaStreamSynchronize(c->st));
    waited = true;
    if (!running()) break;
    ++H.vc_calls;
    RICH_CHECK(fcg_body<T>(c, S, cudaGraphConditionalHandle(0), 0));
    RICH_CUDA(cudaStreamSynchronize(c->st));
  }
  RICH_CUDA(cudaMemcpyAsync(x, k.x, sizeof(double) * n, cudaMemcpyDeviceToDevice, c->st));
  return RICH_OK;
}

// S problems' solves of J x = b from x = 0; per problem the iterations, ||b||, the last
// ||r|| and the reason it stopped (0 converged, else KrylovWork::fail_reason's codes).
// RICH_ENONFINITE if any problem met a non-finite scalar.
int fcg_run(rich_ctx* c, int S, const double* b, double* x, const rich_krylov_opts* o, FcgResult* res) {
  RICH_CHECK(c->prec == RICH_PREC_MIXED ? fcg_solve<float>(c, S, b, x, o) : fcg_solve<double>(c, S, b, x, o));
  const FcgOut* out = static_cast<const FcgOut*>(c->kw.fcg_out);
  int rc = RICH_OK;
  for (int s = 0; s < S; ++s) {
    const int r = out[s].reason;  // 0: the loop left the problem unfinished
    res[s] = FcgResult{out[s].rn, out[s].bn, out[s].it, r == kFcgConverged || r == kFcgZero ? 0 : r ? r : 1};
    if (out[s].reason == kFcgNonfinite) rc = RICH_ENONFINITE;
  }
  return rc;
}

static int fcg(rich_ctx* c, const double* b, double* x, const rich_krylov_opts* o, rich_krylov_stats* st) {
  FcgResult r{};
  const int rc = fcg_run(c, 1, b, x, o, &r);
  st->res0 = r.bn;
  st->res = r.rn;
  st->iterations = r.it;
  st->converged = rc == RICH_OK && r.reason == 0;
  if (rc != RICH_OK) return rc;
  c->kw.fail_reason = r.reason;
  return r.reason == 0 ? RICH_OK : RICH_ENOTCONV_LIN;
}

// V = f src (f = *fdev if given), z = M V.
static int fgmres_precondition(rich_ctx* c, const double* src, const double* fdev, double f, double* V, double* z) {
  const long long n = c->g.n;
  const int g = grid_for(n);
  if (c->H.opts.precond == RICH_PRECOND_AS) {
    k_stage<double><<<g, kBlock, 0, c->st>>>(n, src, fdev, f, V, nullptr, nullptr);
    RICH_LAUNCH_CHECK();
    return as_apply(c, V, z);
  }
  void* b = c->H.lv[0].b;
  const Hierarchy& H = c->H;
  if (c->prec == RICH_PREC_MIXED)
    k_stage<float><<<g, kBlock, 0, c->st>>>(n, src, fdev, f, V, H.scaled ? H.sc32.s : nullptr, (float*)b);
  else
    k_stage<double><<<g, kBlock, 0, c->st>>>(n, src, fdev, f, V, H.scaled ? H.sc64.s : nullptr, (double*)b);
  RICH_LAUNCH_CHECK();
  return vcycle_staged(c, z);
}

// One pass of the orthogonalisation: out = w - V h against nv vectors; h and ||out|| in the
// mirror once the stream has been waited for.
static int gs_pass(rich_ctx* c, int nv, const double* w, double* out) {
  KrylovWork& k = c->kw;
  const long long n = c->g.n;
  const int g = std::min(grid_for(n), kGsBlocks), gu = std::min(grid_for(n, 2 * kBlock), kGsUpdateBlocks);
  {
    ProfScope ps("multidot", c->st, (double)n * 8.0 * (nv + 1), 2.0 * n * nv);  // FP64 operations; G is integer
    k_gs_dots<<<g, kGsThreads, 0, c->st>>>(n, nv, k.V, w, c->partials, k.gram, k.peak, c->ticket, c->dsc, c->hsc);
  }
  RICH_LAUNCH_CHECK();
  {
    ProfScope ps("orth_axpy", c->st, (double)n * 8.0 * (nv + 2), 2.0 * n * (nv + 1));
    k_gs_update<<<gu, kGsThreads, 0, c->st>>>(n, nv, k.V, w, out, c->partials, k.peak + nv, c->ticket, c->dsc, c->hsc);
  }
  RICH_LAUNCH_CHECK();
  return RICH_OK;
}

// Flexible GMRES(m) (Saad) with classical Gram-Schmidt and re-orthogonalisation (gs_pass).
static int fgmres(rich_ctx* c, const double* b, double* x, const rich_krylov_opts* o, rich_krylov_stats* st) {
  KrylovWork& k = c->kw;
  if (!c->H.built) return RICH_ESTATE;
  long long n = c->g.n;
  int m = o->restart;
  int g = grid_for(n);
  double* s = c->dsc;
  RICH_CHECK(nrm2sq(c, b, n, s));
  double h0[1];
  RICH_CHECK(fetch_scalars(c, s, 1, h0));
  double bn = sqrt(h0[0]);
  st->res0 = bn;
  st->res = bn;
  st->iterations = 0;
  st->converged = 0;
  RICH_CUDA(cudaMemsetAsync(x, 0, sizeof(double) * n, c->st));
  if (!std::isfinite(bn)) return RICH_ENONFINITE;
  if (!(bn > 0)) {
    st->converged = 1;
    return RICH_OK;
  }
  double target = o->eta * bn;
  std::vector<double> H((m + 1) * m), cs(m), sn(m), gv(m + 1), y(m);
  auto Hij = [&](int i, int j) -> double& { return H[(size_t)i * m + j]; };
  double beta = bn;
  const double* r0 = b;
  int its = 0;
  for (;;) {
    std::fill(gv.begin(), gv.end(), 0.0);
    gv[0] = beta;
    RICH_CUDA(cudaMemsetAsync(k.peak, 0, sizeof(unsigned), c->st));
    k_gs_peak<<<std::min(grid_for(n), kGsUpdateBlocks), kGsThreads, 0, c->st>>>(n, r0, 1.0 / beta, k.peak);
    RICH_LAUNCH_CHECK();
    int jdone = 0;
    bool conv = false;
    for (int j = 0; j < m; ++j) {
      double* Vj = k.V + (long long)j * n;
      double* Vn = Vj + n;
      double* Zj = k.Z + (long long)j * n;
      // V[j] = r0 / beta, or the last pass's vector over its norm, scaled as it is staged
      RICH_CHECK(j == 0 ? fgmres_precondition(c, r0, nullptr, 1.0 / beta, Vj, Zj)
                        : fgmres_precondition(c, Vj, s + kSlotInv, 0.0, Vj, Zj));
      RICH_CHECK(stencil_apply(c, c->J7, Zj, k.w));
      RICH_CHECK(gs_pass(c, j + 1, k.w, Vn));
      RICH_CUDA(cudaStreamSynchronize(c->st));
      double hn = c->hsc[kSlotNorm], hsq = 0.0;
      for (int i = 0; i <= j; ++i) {
        Hij(i, j) = c->hsc[i];
        hsq += Hij(i, j) * Hij(i, j);
      }
      if (hn * hn < 1e-4 * hsq && hn > 0) {  // cancellation: an explicit projection of what is left
        RICH_CHECK(gs_pass(c, j + 1, Vn, Vn));
        RICH_CUDA(cudaStreamSynchronize(c->st));
        hn = c->hsc[kSlotNorm];
        for (int i = 0; i <= j; ++i) Hij(i, j) += c->hsc[i];
      }
      if (!std::isfinite(hn)) return RICH_ENONFINITE;
      Hij(j + 1, j) = hn;
      for (int i = 0; i < j; ++i) {
        double t = cs[i] * Hij(i, j) + sn[i] * Hij(i + 1, j);
        Hij(i + 1, j) = -sn[i] * Hij(i, j) + cs[i] * Hij(i + 1, j);
        Hij(i, j) = t;
      }
      double den = std::hypot(Hij(j, j), Hij(j + 1, j));
      cs[j] = Hij(j, j) / den;
      sn[j] = Hij(j + 1, j) / den;
      Hij(j, j) = den;
      Hij(j + 1, j) = 0.0;
      gv[j + 1] = -sn[j] * gv[j];
      gv[j] = cs[j] * gv[j];
      ++its;
      jdone = j + 1;
      st->res = fabs(gv[j + 1]);
      if (fabs(gv[j + 1]) <= target || hn == 0.0) {
        conv = true;
        break;
      }
      if (its >= o->maxit) break;
    }
    for (int i = jdone - 1; i >= 0; --i) {
      double acc = gv[i];
      for (int q = i + 1; q < jdone; ++q) acc -= Hij(i, q) * y[q];
      y[i] = acc / Hij(i, i);
    }
    for (int i = 0; i < jdone; ++i) c->hsc[i] = y[i];
    RICH_CUDA(cudaMemcpyAsync(k.hcoef, c->hsc, sizeof(double) * jdone, cudaMemcpyHostToDevice, c->st));
    k_multiaxpy<<<g, kBlock, 0, c->st>>>(n, jdone, k.Z, k.hcoef, 1.0, x);
    RICH_LAUNCH_CHECK();
    st->iterations = its;
    if (conv) {
      st->converged = 1;
      return RICH_OK;
    }
    if (its >= o->maxit) return RICH_ENOTCONV_LIN;
    // restart: r = b - J x
    RICH_CHECK(stencil_apply(c, c->J7, x, k.w));
    k_sub<<<g, kBlock, 0, c->st>>>(n, b, k.w, k.r);
    RICH_LAUNCH_CHECK();
    RICH_CHECK(nrm2sq(c, k.r, n, s));
    RICH_CHECK(fetch_scalars(c, s, 1, h0));
    const double beta_cycle = beta;
    beta = sqrt(h0[0]);
    st->res = beta;
    if (beta <= target) {
      st->converged = 1;
      return RICH_OK;
    }
    if (o->stall > 0 && beta > (1.0 - o->stall) * beta_cycle) {  // the cycle stagnated
      c->kw.fail_reason = 4;
      return RICH_ENOTCONV_LIN;
    }
    r0 = k.r;
  }
}

int krylov_run(rich_ctx* c, const double* b, double* x, const rich_krylov_opts* o, rich_krylov_stats* st) {
  if (o->maxit < 1 || !(o->eta > 0) || !(o->stall >= 0.0 && o->stall < 1.0)) return RICH_EINVAL;
  c->kw.fail_reason = 0;
  if (o->kind == RICH_KRYLOV_FGMRES) {
    if (o->restart < 1 || o->restart > 63) return RICH_EINVAL;
    RICH_CHECK(ensure_krylov(c, o->restart));
    return fgmres(c, b, x, o, st);
  }
  if (o->kind != RICH_KRYLOV_FCG) return RICH_EINVAL;
  RICH_CHECK(ensure_krylov(c, 0));
  return fcg(c, b, x, o, st);
}

// ---------------------------------------------------------------- Newton-Armijo step

static int ensure_newton(rich_ctx* c) {
  if (c->F) return RICH_OK;
  long long n = c->g.n;
  RICH_CHECK(dalloc(&c->s_old, n));
  RICH_CHECK(dalloc(&c->F, n));
  RICH_CHECK(dalloc(&c->Ft, n));
  RICH_CHECK(dalloc(&c->d, n));
  RICH_CHECK(dalloc(&c->ptrial, n));
  RICH_CHECK(dalloc(&c->rhs, n));
  return RICH_OK;
}

// CUDA-event timers of the step's phases; ms accumulate into the target at resolve().
struct PhaseTimers {
  std::vector<cudaEvent_t> ev;
  std::vector<double*> acc;
  std::vector<char> closed;
  cudaStream_t st;
  explicit PhaseTimers(cudaStream_t s) : st(s) {}
  ~PhaseTimers() {
    for (auto e : ev) cudaEventDestroy(e);
  }
  int begin(double* target) {
    int i = (int)acc.size();
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    ev.push_back(a);
    ev.push_back(b);
    acc.push_back(target);
    closed.push_back(0);
    cudaEventRecord(a, st);
    return i;
  }
  void end(int i) {
    cudaEventRecord(ev[2 * i + 1], st);
    closed[i] = 1;
  }
  void resolve() {
    for (size_t i = 0; i < acc.size(); ++i) {
      if (!closed[i]) continue;
      cudaEventSynchronize(ev[2 * i + 1]);
      float t = 0.f;
      cudaEventElapsedTime(&t, ev[2 * i], ev[2 * i + 1]);
      *acc[i] += t;
    }
  }
};

// RAII phase: ends on scope exit, including early error returns.
struct Phase {
  PhaseTimers& pt;
  int i;
  Phase(PhaseTimers& p, double* target) : pt(p), i(p.begin(target)) {}
  ~Phase() { pt.end(i); }
};

static int step_body(rich_ctx* c, double* p, double dt, const rich_newton_opts* o, rich_step_stats* st,
                     PhaseTimers& pt);

static int step_impl(rich_ctx* c, double* p, double dt, const rich_newton_opts* o, rich_step_stats* st) {
  RICH_CHECK(ensure_newton(c));
  long long n = c->g.n;
  int g = grid_for(n);
  memset(st, 0, sizeof(*st));
  st->min_lambda = 1.0;
  PhaseTimers pt(c->st);
  int rc;
  {
    Phase whole(pt, &st->ms_total);
    rc = step_body(c, p, dt, o, st, pt);
  }
  pt.resolve();
  return rc;
}

static int step_body(rich_ctx* c, double* p, double dt, const rich_newton_opts* o, rich_step_stats* st,
                     PhaseTimers& pt) {
  long long n = c->g.n;
  int g = grid_for(n);
  // Converged when ||Phi|| <= max(rtol ||Phi_0||, atol, floor): the floor is
  // eps times the norm of the per-cell magnitudes of the products summed into
  // Phi, the accuracy to which Phi can be evaluated (a step that starts near
  // steady state cannot be driven to rtol ||Phi_0|| below it).
  const double kFloor = 2.220446049250313e-16;
  double h[3];
  {
    Phase ph(pt, &st->ms_feval);
    RICH_CHECK(residual_eval(c, p, nullptr, dt, c->F, true, true, c->s_old));  // s_old = s(p^{l-1})
  }
  RICH_CHECK(wait_scalars(c, 3, h));
  double fn = sqrt(h[0]);
  double floor_ = kFloor * sqrt(h[2]);
  if (!std::isfinite(fn)) return RICH_ENONFINITE;
  st->res0 = st->res = fn;
  double tol = std::max(o->rtol * fn, o->atol);
  for (int r = 0;; ++r) {
    if (fn <= std::max(tol, floor_)) {
      st->converged = 1;
      break;
    }
    if (r == o->max_newton) return RICH_ENOTCONV_NEWTON;
    {
      Phase ph(pt, &st->ms_jacobian);
      // the last residual evaluation was at this p (the start or the accepted trial point)
      RICH_CHECK(jacobian_eval(c, p, dt, true));
    }
    bool rebuild = !c->H.built || (o->amg_policy == RICH_AMG_REBUILD_STEP && r == 0);
    {
      Phase ph(pt, &st->ms_setup);
      if (rebuild) {
        RICH_CHECK(amg_build(c, &o->amg));
        st->amg_setups++;
      } else {
        RICH_CHECK(o->amg_policy == RICH_AMG_SETUP_ONCE ? amg_update_fine(c) : amg_refresh(c));
        st->amg_refreshes++;
      }
    }
    k_scale<<<g, kBlock, 0, c->st>>>(n, c->F, -1.0, c->rhs);
    RICH_LAUNCH_CHECK();
    rich_krylov_stats ks;
    int lin_phase = pt.begin(&st->ms_linsol);
    int s = krylov_run(c, c->rhs, c->d, &o->krylov, &ks);
    st->linear_its += ks.iterations;
    // under time-step control, (p, J p) <= 0 in FCG ends the attempt: the step is retried shorter
    const bool indefinite = o->max_dt_halvings > 0 && c->kw.fail_reason == 2;
    if (s == RICH_ENOTCONV_LIN && o->krylov.kind == RICH_KRYLOV_FCG && !indefinite) {
      rich_krylov_opts fb = o->krylov;
      fb.kind = RICH_KRYLOV_FGMRES;
      fb.restart = o->fcg_fallback_restart;
      st->fallbacks++;
      s = krylov_run(c, c->rhs, c->d, &fb, &ks);
      st->linear_its += ks.iterations;
    }
    pt.end(lin_phase);
    if (s != RICH_OK) return s;
    // slope of f = 1/2 ||Phi||^2 along d: g = Phi . (J d)
    RICH_CHECK(stencil_apply(c, c->J7, c->d, c->Ft));
    RICH_CHECK(dot(c, c->F, c->Ft, n, c->dsc + 2));
    RICH_CHECK(fetch_scalars(c, c->dsc + 2, 1, h));
    double slope = h[0];
    if (!(slope < 0.0)) return RICH_ELINESEARCH;
    double f0 = 0.5 * fn * fn;
    double lam = 1.0, ft = 0.0, floor_t = 0.0;
    for (;;) {
      {
        Phase ph(pt, &st->ms_feval);
        k_axpby<<<g, kBlock, 0, c->st>>>(n, p, lam, c->d, c->ptrial);
        RICH_LAUNCH_CHECK();
        RICH_CHECK(residual_eval(c, c->ptrial, c->s_old, dt, c->Ft, true, true));
      }
      RICH_CHECK(wait_scalars(c, 3, h));
      st->line_search_evals++;
      ft = 0.5 * h[0];
      floor_t = kFloor * sqrt(h[2]);
      if (!std::isfinite(ft)) return RICH_ENONFINITE;
      if (ft <= f0 + o->armijo_c * lam * slope) break;
      double lq = -slope * lam * lam / (2.0 * (ft - f0 - slope * lam));
      lam = std::min(std::max(lq, 0.1 * lam), 0.5 * lam);
      if (lam < o->lambda_min) return RICH_ELINESEARCH;
    }
    RICH_CUDA(cudaMemcpyAsync(p, c->ptrial, sizeof(double) * n, cudaMemcpyDeviceToDevice, c->st));
    std::swap(c->F, c->Ft);
    fn = sqrt(2.0 * ft);
    floor_ = floor_t;
    st->res = fn;
    st->newton_its++;
    st->min_lambda = std::min(st->min_lambda, lam);
  }
  return RICH_OK;
}

// Time-step control: cover dt with backward-Euler substeps of length dt / 2^k.  A
// substep that fails to converge is discarded (p restored) and retried with half
// its length, down to dt / 2^H; after an accepted substep the length doubles back
// whenever the time reached (counted in units of dt / 2^H) is a multiple of the
// doubled length, so the substeps end exactly at dt.
// A Krylov solve that merely ran out of iterations ends the step: a shorter step
// does not mend the preconditioner, and retrying would multiply the cost.  FCG's
// (p, J p) <= 0 on an indefinite Jacobian is retried.
static bool retryable(rich_ctx* c, int s) {
  if (s == RICH_ENOTCONV_NEWTON || s == RICH_ELINESEARCH) return true;
  return s == RICH_ENOTCONV_LIN && c->kw.fail_reason == 2;
}

static int advance_impl(rich_ctx* c, double* p, double dt, const rich_newton_opts* o, rich_step_stats* st) {
  const int H = o->max_dt_halvings;
  if (H > 40) return RICH_EINVAL;
  long long n = c->g.n;
  if (!c->psave) RICH_CHECK(dalloc(&c->psave, n));
  memset(st, 0, sizeof(*st));
  st->min_lambda = 1.0;
  st->dt_min = dt;
  const long long total = 1LL << H;
  long long t = 0;
  int k = 0;
  bool first = true;
  while (t < total) {
    const double h = std::ldexp(dt, -k);
    const long long len = 1LL << (H - k);
    RICH_CUDA(cudaMemcpyAsync(c->psave, p, sizeof(double) * n, cudaMemcpyDeviceToDevice, c->st));
    rich_step_stats sub;
    int s = step_impl(c, p, h, o, &sub);
    st->newton_its += sub.newton_its;
    st->linear_its += sub.linear_its;
    st->line_search_evals += sub.line_search_evals;
    st->fallbacks += sub.fallbacks;
    st->amg_setups += sub.amg_setups;
    st->amg_refreshes += sub.amg_refreshes;
    st->ms_feval += sub.ms_feval;
    st->ms_jacobian += sub.ms_jacobian;
    st->ms_setup += sub.ms_setup;
    st->ms_linsol += sub.ms_linsol;
    st->ms_total += sub.ms_total;
    if (first) st->res0 = sub.res0;
    first = false;
    st->res = sub.res;
    if (s != RICH_OK) {
      if (s != RICH_ECUDA)  // the substep's start is the last accepted state
        RICH_CUDA(cudaMemcpyAsync(p, c->psave, sizeof(double) * n, cudaMemcpyDeviceToDevice, c->st));
      if (!retryable(c, s)) return s;
      st->dt_failures++;
      if (k == H) return s;
      ++k;
      continue;
    }
    st->min_lambda = std::min(st->min_lambda, sub.min_lambda);
    t += len;
    st->substeps++;
    st->dt_min = std::min(st->dt_min, h);
    if (k > 0 && t % (2 * len) == 0) --k;
  }
  st->converged = 1;
  return RICH_OK;
}

}  // namespace rich

using namespace rich;

extern "C" {

int amg_vcycle(rich_ctx* c, const double* r, double* z) {
  if (!c || !r || !z) return RICH_EINVAL;
  AllocStream guard(c->st);
  return vcycle_apply(c, r, z);
}

int krylov_solve(rich_ctx* c, const double* b, double* x, const rich_krylov_opts* o, rich_krylov_stats* st) {
  if (!c || !b || !x || !o) return RICH_EINVAL;
  AllocStream guard(c->st);
  if (!c->have_jac || !c->H.built) return RICH_ESTATE;
  rich_krylov_stats tmp;
  return krylov_run(c, b, x, o, st ? st : &tmp);
}

int rich_step(rich_ctx* c, double* p, double dt, const rich_newton_opts* o, rich_step_stats* st) {
  if (!c || !p || !(dt > 0)) return RICH_EINVAL;
  AllocStream guard(c->st);
  rich_newton_opts def;
  if (!o) {
    rich_default_newton_opts(&def);
    o = &def;
  }
  rich_step_stats tmp;
  if (!st) st = &tmp;
  if (o->max_dt_halvings < 0) return RICH_EINVAL;
  if (o->max_dt_halvings > 0) return advance_impl(c, p, dt, o, st);
  int s = step_impl(c, p, dt, o, st);
  st->substeps = s == RICH_OK ? 1 : 0;
  st->dt_min = dt;
  return s;
}

int rich_step_host(rich_ctx* c, double* p_host, double dt, const rich_newton_opts* o, rich_step_stats* st) {
  if (!c || !p_host || !(dt > 0)) return RICH_EINVAL;
  AllocStream guard(c->st);
  long long n = c->g.n;
  if (!c->pbuf) RICH_CHECK(dalloc(&c->pbuf, n));
  RICH_CUDA(cudaMemcpyAsync(c->pbuf, p_host, sizeof(double) * n, cudaMemcpyHostToDevice, c->st));
  int s = rich_step(c, c->pbuf, dt, o, st);
  RICH_CUDA(cudaMemcpyAsync(p_host, c->pbuf, sizeof(double) * n, cudaMemcpyDeviceToHost, c->st));
  RICH_CUDA(cudaStreamSynchronize(c->st));
  return s;
}

}  // extern "C"

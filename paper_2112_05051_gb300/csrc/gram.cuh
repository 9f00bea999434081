// Gram-Schmidt of FGMRES, in two passes over the basis (classical Gram-Schmidt with
// the second projection taken from the basis' Gram matrix: Swirydowicz, Langou, Ananthan,
// Yang, Thomas, "Low synchronization Gram-Schmidt and generalized minimal residual
// algorithms", 2021).  With G = V^T V, whose last row is the new vector's dots, the
// coefficients of two projections are h = h1 + (I - G) h1, h1 = V^T w, so the basis is read
// once for the dots (with w and with the newest vector) and once for w - V h.  h's rounding
// is relative to ||w||, so each vector is orthogonal to those before it to ||w|| / ||w - V h||
// units; where that passes a hundred (||w - V h|| < 1e-2 ||h||) the host asks for one explicit
// pass more.  A numpy model, 30 vectors: ||V^T V - I|| 2e-14 where 0.3 of w is left, 5e-13 just
// above 0.01, against 1e-15 with two explicit projections.  The solve does not feel it:
// J Z = V H holds to rounding for whatever h is subtracted, and ||V t|| is ||t|| to that 5e-13.
// Solves to 1e-7 ... 1e-15 (68 x 65 x 4 to 64^3 cells) take the same iterations, and leave the
// same true residuals, as with two explicit projections.
// Bound: the FP64 pipe, two operations per basis element, one in either pass (explicit second
// projections take four and read the basis four times), and in the dots the loads.
// 128^3, FGMRES(30): 667 us per iteration with two explicit projections, 545 with a Gram matrix
// summed in FP64, 518 with one summed in integers (dots at ten vectors: 101 -> 75 us).
#pragma once

#include "common.cuh"

namespace rich {

constexpr int kGsThreads = 256;
// Of the dots: one wave at 80 registers (4 per SM with 64 registers: 93 us against 83).
constexpr int kGsBlocks = 3 * kNumSM;
constexpr int kGsUpdateBlocks = 4 * kNumSM;  // of the update: one wave (8 per SM left a second, 59 us against 46)
constexpr int kGsTile = 4;             // basis vectors per sweep over a block's elements
constexpr int kGsLd = 64;              // row length of the Gram matrix
// Device scalars of an iteration (restart <= 63): h in [0, j], ||w - V h|| and its reciprocal.
constexpr int kSlotNorm = 63, kSlotInv = 64;

// Sums of 8 values over a warp by halving: after the exchange at distances 16, 8 and 4 a
// lane holds one value, summed on at 2 and 1: 9 additions instead of 40.  The lane's value
// is number lane >> 2.
__device__ __forceinline__ double warp_sum8(double (&a)[8]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 4; k > 0; k >>= 1) {
    const bool up = lane & (4 * k);
#pragma unroll
    for (int q = 0; q < k; ++q) {
      const double keep = up ? a[q + k] : a[q], send = up ? a[q] : a[q + k];
      a[q] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * k);
    }
  }
  a[0] += __shfl_xor_sync(0xffffffffu, a[0], 2);
  a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
  return a[0];
}

// G's entries are summed in integers, in units of a power of two that follows each vector's
// largest entry.  With 2^(top - 1023) above every |v|, an entry in units of 2^(top - 1083) is
// h 2^30 + l with |h| <= 2^30 and |l| <= 2^29, and a product is four 32-bit multiply-adds into
// three 64-bit sums; those and the split (20 integer instructions) run beside the FP64 pipe,
// which is left with the dots with w alone.  An entry's rounding, half a unit, is all that
// the integers lose, and like entries lose alike: G_ab is off by up to u_a ||b||_1 + u_b ||a||_1
// (u half the units).  A spread vector of n cells has a largest entry near n^-1/2, which
// makes that about 2^-58 for every n (in units of 2^-60 for all vectors it was 2^-60 n^1/2,
// measured 3.8e-15 for a constant of 16M cells); under a single large entry a tail keeps
// units of 2^-60.  |G - V^T V| measured on constant, smooth, random and one-sided vectors of
// 1e3 to 1.6e7 cells 4.4e-16 at most, with a single large entry 6.7e-16, on the bases of 128^3
// and 399 x 401 x 19 solves 2.2e-16; torch's FP64 dots of the same: 2.2e-16, 7.8e-16 and 2.2e-16.
struct UnitFixed {
  int h, l;
};
// top for a vector whose largest |v| has the high word hi (read as unsigned): h of per-thread
// sums of m products may not pass 2^60, so the unit leaves c = ceil(log2(m) / 2) bits over it;
// 1023 at most, which serves every vector of norm 1 (the sum of all h^2 is 2^60 then).
__device__ __forceinline__ unsigned unit_top(unsigned hi, long long m) {
  const int c = m > 1 ? (65 - __clzll(m - 1)) / 2 : 0;
  return (unsigned)min(max((int)(hi >> 20) + 1 + c, 1023 - 40), 1023);
}
__device__ __forceinline__ UnitFixed unit_fixed(double v, unsigned top) {
  const int hi = __double2hiint(v), sg = hi >> 31;
  const unsigned e = ((unsigned)hi >> 20) & 0x7ffu, s = min(top - e, 63u);
  // twice the magnitude in units, shifted, then rounded to nearest
  unsigned long long m = (unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32;
  m |= (unsigned)__double2loint(v);
  m = (((m << 9) >> s) + 1) >> 1;
  const int h = (int)((m + (1u << 29)) >> 30), l = (int)((unsigned)m - ((unsigned)h << 30));
  return {(h ^ sg) - sg, (l ^ sg) - sg};
}
// Sums of products: hh 2^-60 + x 2^-90 + ll 2^-120 (in the vectors' scales), carried after
// every kUnitRun of them.  |ll| grows by 2^58 a product; |x| stays below 2 2^29 sqrt(16) 2^30
// and |hh| below 2^60 because sum h^2 <= 2^60 over a thread's share of a vector (unit_top).
constexpr int kUnitRun = 16;
struct UnitSum {
  long long hh = 0, x = 0, ll = 0;
  __device__ __forceinline__ void add(UnitFixed a, UnitFixed b) {
    hh += (long long)a.h * b.h;
    x += (long long)a.h * b.l;
    x += (long long)a.l * b.h;
    ll += (long long)a.l * b.l;
  }
  __device__ __forceinline__ void carry() {
    x += ll >> 30;
    ll &= (1 << 30) - 1;
    hh += x >> 30;
    x &= (1 << 30) - 1;
  }
  // The sum in units of 2^-60, with one conversion of its leading 61 bits (rounded to a fixed
  // unit of 2^-62, a constant's equal sums were off by 116736 times the same remainder:
  // 9e-15 for 300k cells).
  __device__ __forceinline__ double value() {
    carry();
    const int k = min(__clzll(hh ^ (hh >> 63)) - 2, 30);  // hh 2^k below 2^62
    const long long r = k < 30 ? 1LL << (29 - k) : 0;
    const long long t = (long long)((unsigned long long)hh << k) + ((x + r) >> (30 - k));
    const double v = (double)t;  // 0 or at least 1: its exponent takes the 2^-k
    return __hiloint2double(__double2hiint(v) - (t ? k << 20 : 0), __double2loint(v));
  }
};

// Copies of 8 bytes into the thread's own words of shared memory, kGsStages elements deep:
// the loads of the next elements run under this one's arithmetic and hold no registers
// (with plain loads the warps waited for memory two thirds of the time: 147 us, ten vectors).
constexpr int kGsStages = 3;
typedef double GsStage[kGsTile + 2][kGsThreads];
__device__ __forceinline__ void copy8(double* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// The block's sums over its elements of M basis vectors (from v0) times w and vj, into
// a[q] and a[4 + q].  tops: the nv vectors' unit_top, filled here for the first sweep (the
// loads are under way by then) from this thread's vector's peak.
template <int M>
__device__ __forceinline__ void gs_tile(long long n, const double* v0, const double* w, const double* vj,
                                        unsigned* tops, int q0, int nv, unsigned peak, GsStage (&st)[kGsStages],
                                        double (&a)[8]) {
  const long long stride = (long long)gridDim.x * kGsThreads;
  const int t = threadIdx.x;
  auto fetch = [&](int slot, long long i) {
    if (i < n) {
#pragma unroll
      for (int q = 0; q < M; ++q) copy8(&st[slot][q][t], v0 + q * n + i);
      copy8(&st[slot][kGsTile][t], w + i);
      copy8(&st[slot][kGsTile + 1][t], vj + i);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  long long i = blockIdx.x * (long long)kGsThreads + t;
#pragma unroll
  for (int k = 0; k < kGsStages; ++k) fetch(k, i + k * stride);
  if (q0 == 0) {
    if (t < nv) tops[t] = unit_top(peak, (n + stride - 1) / stride);
    __syncthreads();
  }
  UnitSum g[M];
  unsigned top[M];
  const unsigned topj = tops[nv - 1];
#pragma unroll
  for (int q = 0; q < M; ++q) top[q] = tops[q0 + q];
  int run = 0, slot = 0;
#pragma unroll 1
  for (; i < n; i += stride) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kGsStages - 1) : "memory");
    double p[M];
    const double w0 = st[slot][kGsTile][t], x0 = st[slot][kGsTile + 1][t];
#pragma unroll
    for (int q = 0; q < M; ++q) p[q] = st[slot][q][t];
    const UnitFixed f = unit_fixed(x0, topj);
#pragma unroll
    for (int q = 0; q < M; ++q) {
      a[q] = fma(p[q], w0, a[q]);
      g[q].add(unit_fixed(p[q], top[q]), f);
    }
    if (++run == kUnitRun) {
#pragma unroll
      for (int q = 0; q < M; ++q) g[q].carry();
      run = 0;
    }
    fetch(slot, i + kGsStages * stride);  // into the words just read
    slot = slot == kGsStages - 1 ? 0 : slot + 1;
  }
#pragma unroll
  for (int q = 0; q < M; ++q) a[4 + q] = g[q].value();
}

// h1 = V^T w and the newest row of G = V^T V (nv vectors, vj = V[nv - 1]); the last block
// to finish forms h and leaves it at s[0, nv) and in the pinned mirror.
__global__ void __launch_bounds__(kGsThreads, 3) k_gs_dots(long long n, int nv, const double* __restrict__ V,
                                                        const double* __restrict__ w, double* __restrict__ part,
                                                        double* __restrict__ gram, const unsigned* __restrict__ peak,
                                                        unsigned* __restrict__ ticket, double* __restrict__ s,
                                                        double* __restrict__ mirror) {
  constexpr int W = kGsThreads / 32;
  __shared__ double sh[W][2 * kGsTile];
  __shared__ double tot[2 * kGsLd];
  __shared__ GsStage st[kGsStages];
  __shared__ bool last;
  const double* vj = V + (long long)(nv - 1) * n;
  __shared__ unsigned tops[kGsLd];
  const unsigned own = threadIdx.x < nv ? peak[threadIdx.x] : 0;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int q0 = 0; q0 < nv; q0 += kGsTile) {
    double a[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const double* v0 = V + (long long)q0 * n;
    const int m = min(kGsTile, nv - q0);
    if (m == 4) gs_tile<4>(n, v0, w, vj, tops, q0, nv, own, st, a);
    else if (m == 3) gs_tile<3>(n, v0, w, vj, tops, q0, nv, own, st, a);
    else if (m == 2) gs_tile<2>(n, v0, w, vj, tops, q0, nv, own, st, a);
    else gs_tile<1>(n, v0, w, vj, tops, q0, nv, own, st, a);
    const double r = warp_sum8(a);
    if ((lane & 3) == 0) sh[wid][lane >> 2] = r;
    __syncthreads();
    if (threadIdx.x < 8 && (threadIdx.x & 3) < m) {
      double t = 0.0;
      for (int k = 0; k < W; ++k) t += sh[k][threadIdx.x];
      const int q = (threadIdx.x >> 2) * kGsLd + q0 + (threadIdx.x & 3);
      part[(long long)q * gridDim.x + blockIdx.x] = t;
    }
    __syncthreads();
  }
  if (threadIdx.x < 8) __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int t = wid; t < 2 * nv; t += W) {
    const int q = t < nv ? t : kGsLd + t - nv;
    double a = 0.0;
    for (int k = lane; k < (int)gridDim.x; k += 32) a += __ldcg(&part[(long long)q * gridDim.x + k]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    if (lane == 0) {
      if (t >= nv) {  // from the integers' units
        const int k = 60 + 2 * 1023 - (int)tops[t - nv] - (int)tops[nv - 1];
        a *= __hiloint2double((1023 - k) << 20, 0);
      }
      tot[q] = a;
    }
  }
  __syncthreads();
  if (threadIdx.x < nv)
    gram[(nv - 1) * kGsLd + threadIdx.x] = gram[threadIdx.x * kGsLd + nv - 1] = tot[kGsLd + threadIdx.x];
  __syncthreads();
  for (int i = wid; i < nv; i += W) {  // h_i = h1_i + sum_q (I - G)_iq h1_q
    double d = 0.0;
    for (int q = lane; q < nv; q += 32) d = fma((q == i ? 1.0 : 0.0) - gram[i * kGsLd + q], tot[q], d);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
    if (lane == 0) s[i] = mirror[i] = tot[i] + d;
  }
  if (threadIdx.x == 0) *ticket = 0;
}

__device__ __forceinline__ unsigned abs_hi(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

// *peak, zero before: the high word of the largest |f v|, for a cycle's first vector.
__global__ void __launch_bounds__(kGsThreads) k_gs_peak(long long n, const double* __restrict__ v, double f,
                                                        unsigned* __restrict__ peak) {
  unsigned hi = 0;
  for (long long i = blockIdx.x * (long long)kGsThreads + threadIdx.x; i < n; i += (long long)gridDim.x * kGsThreads)
    hi = max(hi, abs_hi(f * v[i]));
  hi = __reduce_max_sync(0xffffffffu, hi);
  if ((threadIdx.x & 31) == 0 && hi > __ldcg(peak)) atomicMax(peak, hi);
}

// out = w - V h (w may be out) and its norm: the last block leaves ||out|| and 1/||out||
// (0 for a zero vector) in the scalars, the norm in the mirror, and in *peak (the next
// vector's) the high word of the largest |out| / ||out||, or one more.
__global__ void __launch_bounds__(kGsThreads) k_gs_update(long long n, int nv, const double* __restrict__ V,
                                                          const double* w, double* out, double* __restrict__ part,
                                                          unsigned* __restrict__ peak, unsigned* __restrict__ ticket,
                                                          double* __restrict__ s, double* __restrict__ mirror) {
  __shared__ double hs[kGsLd];
  __shared__ bool last;
  __shared__ unsigned big[2];  // largest high words, of the block and of all
  if (threadIdx.x < 2) big[threadIdx.x] = 0;
  for (int q = threadIdx.x; q < nv; q += kGsThreads) hs[q] = s[q];
  __syncthreads();
  const long long stride = (long long)gridDim.x * kGsThreads;
  double acc[1] = {0.0};
  unsigned hi = 0;
  long long i = blockIdx.x * (long long)kGsThreads + threadIdx.x;
  for (; i + stride < n; i += 2 * stride) {
    double t = w[i], u = w[i + stride];
    const double* v = V + i;
#pragma unroll 4
    for (int q = 0; q < nv; ++q, v += n) {
      t = fma(-hs[q], v[0], t);
      u = fma(-hs[q], v[stride], u);
    }
    out[i] = t;
    out[i + stride] = u;
    acc[0] = fma(t, t, acc[0]);
    acc[0] = fma(u, u, acc[0]);
    hi = max(hi, max(abs_hi(t), abs_hi(u)));
  }
  if (i < n) {
    double t = w[i];
#pragma unroll 4
    for (int q = 0; q < nv; ++q) t = fma(-hs[q], V[(long long)q * n + i], t);
    out[i] = t;
    acc[0] = fma(t, t, acc[0]);
    hi = max(hi, abs_hi(t));
  }
  hi = __reduce_max_sync(0xffffffffu, hi);
  if ((threadIdx.x & 31) == 0) atomicMax(&big[0], hi);
  block_sum<1>(acc);  // (its barriers order big, too)
  if (threadIdx.x == 0) {
    part[blockIdx.x] = acc[0];
    part[gridDim.x + blockIdx.x] = __hiloint2double((int)big[0], 0);
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  acc[0] = 0.0;
  hi = 0;
  for (int k = threadIdx.x; k < (int)gridDim.x; k += kGsThreads) {
    acc[0] += __ldcg(&part[k]);
    hi = max(hi, abs_hi(__ldcg(&part[gridDim.x + k])));
  }
  hi = __reduce_max_sync(0xffffffffu, hi);
  if ((threadIdx.x & 31) == 0) atomicMax(&big[1], hi);
  block_sum<1>(acc);
  if (threadIdx.x == 0) {
    const double h = sqrt(acc[0]), inv = h > 0 ? 1.0 / h : 0.0;
    s[kSlotNorm] = mirror[kSlotNorm] = h;
    s[kSlotInv] = inv;
    *peak = abs_hi(__hiloint2double((int)big[1], -1) * inv);
    *ticket = 0;
  }
}

// V = f src (f from the device if fdev), and the V-cycle's right-hand side with it (scaled
// by sc, if given).
template <class T>
__global__ void k_stage(long long n, const double* src, const double* __restrict__ fdev, double f, double* V,
                        const T* __restrict__ sc, T* __restrict__ b) {
  if (fdev) f = *fdev;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double v = f * src[i];
    V[i] = v;
    if (b) b[i] = sc ? sc[i] * (T)v : (T)v;
  }
}

}  // namespace rich

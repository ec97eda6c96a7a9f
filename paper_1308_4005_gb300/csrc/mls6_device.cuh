// Device helpers shared by the kernels of the multilevel summation library.
#pragma once
#include <climits>

#include <cuda_runtime.h>

#include "mls6_internal.h"

namespace mls6 {

// Block coordinates of a kernel body: the hardware block index and grid
// size in a kernel of its own, a work item's block index and block count
// when a persistent kernel runs the body.
struct Blk {
  unsigned x, n;
  static __device__ __forceinline__ Blk self() { return Blk{blockIdx.x, gridDim.x}; }
};

template <typename T> struct Box3 {
  T L[3], invL[3];
};

// i mod n in [0, n).  Indices are nearly always within one period of the
// grid (a node's neighbours), which is tested first; the remainder is taken
// only for grids narrower than the offset (repeated wrapping).
__device__ __forceinline__ int wrapi(int i, int n) {
  if ((unsigned)i < (unsigned)n) return i;
  if (i < 0 && i >= -n) return i + n;
  if (i >= n && i - n < n) return i - n;
  const int m = i % n;
  return m < 0 ? m + n : m;
}

// Position wrapped into [0, L).
template <typename T> __device__ __forceinline__ T wrapx(T x, T L, T invL) {
  T r = x - floor(x * invL) * L;
  if (r < T(0)) r += L;
  if (r >= L) r -= L;
  if (!(r >= T(0) && r < L)) r = T(0);
  return r;
}

// Weights of the four nodes base-1 .. base+2 of Eq. (Phi-Hermite) for an
// atom at fractional offset t in [0,1) from node base -- Phi(1+t), Phi(t),
// Phi(1-t), Phi(2-t) -- and (phi4 only) their derivatives in t.
template <typename T> __device__ __forceinline__ void phi4w(T t, T w[4]) {
  T s = T(1) - t;
  w[0] = T(-0.5) * t * s * s;
  w[1] = s * (T(1) + t - T(1.5) * t * t);
  w[2] = t * (T(1) + s - T(1.5) * s * s);
  w[3] = T(-0.5) * s * t * t;
}

template <typename T> __device__ __forceinline__ void phi4(T t, T w[4], T dw[4]) {
  phi4w(t, w);
  T s = T(1) - t;
  dw[0] = T(-0.5) * s * (T(1) - T(3) * t);
  dw[1] = t * (T(-5) + T(4.5) * t);
  dw[2] = s * (T(5) - T(4.5) * s);
  dw[3] = T(-0.5) * t * (T(2) - T(3) * t);
}

// Order p = 5: the C^1 quintic (even, support |t| < 3, reproducing
// polynomials of degree <= 4; the member whose outer piece continues to a
// root at |t| = 4).  Weights of the six nodes base-2 .. base+3 of an atom at
// offset t in [0,1) from node base -- Phi(2+t), Phi(1+t), Phi(t), Phi(1-t),
// Phi(2-t), Phi(3-t) -- in factored form (no cancellation near the ends of
// the support), and (phi6 only) their derivatives in t.
template <typename T> __device__ __forceinline__ void phi6w(T t, T w[6]) {
  const T s = T(1) - t, tp = T(1) + t, tm = T(2) - t;
  const T k24 = T(1.0 / 24.0), k12 = T(1.0 / 12.0);
  w[0] = k24 * t * s * s * tp * tm;
  w[1] = k24 * t * s * tm * (T(5) * t * t + t - T(8));
  w[2] = k12 * s * tm * tp * (T(6) + T(3) * t - T(5) * t * t);
  w[3] = k12 * t * tm * tp * (T(4) + T(7) * t - T(5) * t * t);
  w[4] = k24 * t * s * tp * (T(5) * t * t - T(11) * t - T(2));
  w[5] = k24 * t * t * s * tm * tp;
}

template <typename T> __device__ __forceinline__ void phi6(T t, T w[6], T dw[6]) {
  phi6w(t, w);
  const T s = T(1) - t;
  const T k24 = T(1.0 / 24.0), k12 = T(1.0 / 12.0);
  dw[0] = k24 * s * (((T(5) * t - T(7)) * t - T(4)) * t + T(2));
  dw[1] = k24 * ((((T(25) * t - T(56)) * t - T(3)) * t + T(52)) * t - T(16));
  dw[2] = -k12 * t * (((T(25) * t - T(52)) * t - T(15)) * t + T(50));
  dw[3] = -k12 * s * (((T(25) * t - T(23)) * t - T(44)) * t - T(8));
  dw[4] = -k24 * ((((T(25) * t - T(44)) * t - T(21)) * t + T(22)) * t + T(2));
  dw[5] = k24 * t * (((T(5) * t - T(8)) * t - T(3)) * t + T(4));
}

// Basis of NP = p + 1 nodes per axis: weights (and derivatives) of nodes
// base - (NP/2 - 1) .. base + NP/2.
template <int NP, typename T> __device__ __forceinline__ void phiw(T t, T* w) {
  if constexpr (NP == 6)
    phi6w(t, w);
  else
    phi4w(t, w);
}
template <int NP, typename T> __device__ __forceinline__ void phid(T t, T* w, T* dw) {
  if constexpr (NP == 6)
    phi6(t, w, dw);
  else
    phi4(t, w, dw);
}

// Restriction / prolongation: Phi at half-integers.  For a fine node at
// coarse position c + 1/2 the NP coarse nodes c - (NP/2 - 1) .. c + NP/2
// weigh Phi(NP/2 - 1/2), ..., Phi(1/2), Phi(1/2), ..., Phi(NP/2 - 1/2);
// restriction takes the same values at fine offsets +-1, +-3, +-5 from 2 mu.
template <int NP, typename T> __device__ __forceinline__ T half_weight(int k) {
  // k = 0: Phi(1/2), 1: Phi(3/2), 2: Phi(5/2)
  if constexpr (NP == 6)
    return k == 0 ? T(150.0 / 256.0) : (k == 1 ? T(-25.0 / 256.0) : T(3.0 / 256.0));
  else
    return k == 0 ? T(0.5625) : T(-0.0625);
}

// Programmatic dependent launch: every kernel of the evaluation chain first
// waits until its predecessor has completed and flushed (wait), then lets
// its successor be scheduled (launch_dependents), so the successor's launch
// overlaps this kernel's work while every memory access still follows plain
// stream order.  Triggering before the wait let whole chains of waiting
// kernels become resident at once, and under CUDA-graph replay a kernel
// then read a value (the fixed-point scale) that two launches earlier had
// not yet written; with the trigger after the wait at most one kernel waits
// ahead of the running one.  Both are no-ops for a kernel launched without
// the programmatic-serialization attribute.
//
// The wait orders memory operations only for the compiler's ordinary loads:
// a load through a `const T* __restrict__` parameter is treated as
// invariant for the whole kernel and may be scheduled above the wait.
// pdl_begin therefore returns a zero produced by an opaque instruction after
// the wait; kernels add it to every such pointer (`p += z`), so no load
// through them can be issued before the wait (the pointers stay based on
// their restrict parameters).
__device__ __forceinline__ long pdl_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  long z;
  asm volatile("mov.b64 %0, 0;" : "=l"(z)::"memory");
  return z;
}

// ------------------------------------------------- work queues of persistent kernels

struct PQueue {
  unsigned long long ticket;  // next item
  int error;                  // bit 0: a bounded wait ran out
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// ------------------------------------------------- nodes around a block's atoms

// A block of consecutive cell-sorted atoms touches a compact box of grid
// nodes.  Where that box fits into kNodeBoxBytes, the block keeps it in shared
// memory: the anterpolation sums there, the features read there.  One buffer
// per kernel, whatever stages it runs; in the persistent kernel the start of
// its dynamic shared memory, of which the transforms take up to 200 KB (beside
// 24 KB of static memory that is more than a block may have).
constexpr int kNodeBoxBytes = 24 * 1024;
#ifdef MLS6_DEVICE_ONLY
extern __shared__ __align__(16) unsigned char persist_smem[];
__device__ __forceinline__ unsigned char* node_box_smem() { return persist_smem; }
#else
__device__ __forceinline__ unsigned char* node_box_smem() {
  __shared__ __align__(16) unsigned char buf[kNodeBoxBytes];
  return buf;
}
#endif

// Unwrapped node indices lo .. lo + e - 1 per axis; in: the box fits and every
// index is at most one period away from its node (the same for all threads).
struct NodeBox {
  int lo0, lo1, lo2, e0, e1, e2;
  bool in;
};

// Box of the nodes b - BELOW .. b + ABOVE of the block's valid atoms.
template <int BELOW, int ABOVE>
__device__ __forceinline__ NodeBox block_node_box(bool valid, int b0, int b1, int b2, int n0,
                                                  int n1, int n2, int cap) {
  __shared__ int lim[6];
  if (threadIdx.x < 6) lim[threadIdx.x] = threadIdx.x < 3 ? INT_MAX : INT_MIN;
  __syncthreads();
  const int l0 = __reduce_min_sync(0xffffffffu, valid ? b0 - BELOW : INT_MAX);
  const int l1 = __reduce_min_sync(0xffffffffu, valid ? b1 - BELOW : INT_MAX);
  const int l2 = __reduce_min_sync(0xffffffffu, valid ? b2 - BELOW : INT_MAX);
  const int h0 = __reduce_max_sync(0xffffffffu, valid ? b0 + ABOVE : INT_MIN);
  const int h1 = __reduce_max_sync(0xffffffffu, valid ? b1 + ABOVE : INT_MIN);
  const int h2 = __reduce_max_sync(0xffffffffu, valid ? b2 + ABOVE : INT_MIN);
  if ((threadIdx.x & 31) == 0 && l0 != INT_MAX) {
    atomicMin(&lim[0], l0);
    atomicMin(&lim[1], l1);
    atomicMin(&lim[2], l2);
    atomicMax(&lim[3], h0);
    atomicMax(&lim[4], h1);
    atomicMax(&lim[5], h2);
  }
  __syncthreads();
  NodeBox B;
  B.lo0 = lim[0];
  B.lo1 = lim[1];
  B.lo2 = lim[2];
  B.in = lim[3] >= lim[0] && min(n0, min(n1, n2)) > max(BELOW, ABOVE);
  B.e0 = B.in ? lim[3] - lim[0] + 1 : 0;
  B.e1 = B.in ? lim[4] - lim[1] + 1 : 0;
  B.e2 = B.in ? lim[5] - lim[2] + 1 : 0;
  B.in = B.in && (long)B.e0 * B.e1 * B.e2 <= cap;
  return B;
}

// Index at most one period outside [0, n).
__device__ __forceinline__ int wrap1(int i, int n) {
  i += i < 0 ? n : 0;
  return i - (i >= n ? n : 0);
}

// The box's node values, x fastest: one warp per row, asynchronous copies.
template <typename T>
__device__ __forceinline__ void load_node_box(T* box, const T* __restrict__ src, const NodeBox& B,
                                              int n0, int n1, int n2) {
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int r = threadIdx.x >> 5; r < B.e1 * B.e2; r += nw) {
    const int c = r / B.e1, b = r - c * B.e1;
    const T* row = src + (long)n0 * (wrap1(B.lo1 + b, n1) + (long)n1 * wrap1(B.lo2 + c, n2));
    const unsigned dst = (unsigned)__cvta_generic_to_shared(box + r * B.e0);
    for (int x = lane; x < B.e0; x += 32)
      asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(
                       dst + x * (unsigned)sizeof(T)),
                   "l"(row + wrap1(B.lo0 + x, n0)), "n"(sizeof(T))
                   : "memory");
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// *w = max(*w, v); most blocks find it reached already, which spares them the
// atomic (thousands on one word take microseconds).
template <typename I> __device__ __forceinline__ void raise_to(I* w, I v) {
  if (*(volatile I*)w < v) atomicMax(w, v);
}

// Least and largest over the warp of values >= 0 (FP32: their bits order like
// unsigned integers, one instruction each instead of five exchanges).
__device__ __forceinline__ void warp_range(float& lo, float& hi) {
  lo = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(lo)));
  hi = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(hi)));
}
__device__ __forceinline__ void warp_range(double& lo, double& hi) {
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
}

// Sums over a warp of NV = 5..8 values per lane: lane l returns the sum of
// value l / 4.  Halves of the values are exchanged, so that a lane adds
// 4 + 2 + 1 + 1 + 1 times instead of 5 NV times; every sum is the same tree as
// NV separate shuffle reductions, bit for bit.  In FP64, at 2 lanes per cycle
// and SM, seven sums over a block of 256 took 2.4 us of issue.
template <typename T, int NV>
__device__ __forceinline__ T warp_sums(const T (&v)[NV]) {
  static_assert(NV > 4 && NV <= 8, "");
  const int lane = threadIdx.x & 31;
  T a[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) a[c] = c < NV ? v[c < NV ? c : 0] : T(0);
#pragma unroll
  for (int h = 4, o = 16; h > 0; h >>= 1, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const T keep = up ? a[h + k] : a[k], send = up ? a[k] : a[h + k];
      a[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  a[0] += __shfl_xor_sync(0xffffffffu, a[0], 2);
  return a[0] + __shfl_xor_sync(0xffffffffu, a[0], 1);
}

// Second step of the block sums: warp 0 adds the warps' sums sh[c * 32 + warp]
// in order, one lane per value.
template <int NV> __device__ __forceinline__ void add_warps(double (&out)[NV], const double* sh) {
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (threadIdx.x >= 32) return;
  double s = 0.0;
  if (lane < NV)
    for (int w = 0; w < nw; ++w) s += sh[lane * 32 + w];
#pragma unroll
  for (int c = 0; c < NV; ++c) out[c] = __shfl_sync(0xffffffffu, s, c);
}

// Block-wide sums of NV doubles (blockDim.x a multiple of 32, <= 1024);
// results valid in thread 0; fixed reduction order.  sh: >= 32*NV doubles.
template <int NV> __device__ __forceinline__ void block_sum_n(double (&v)[NV], double* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if constexpr (NV > 4) {
    const double t = warp_sums(v);
    __syncthreads();
    if ((lane & 3) == 0 && (lane >> 2) < NV) sh[(lane >> 2) * 32 + wid] = t;
  } else {
#pragma unroll
    for (int c = 0; c < NV; ++c) v[c] = warp_sum(v[c]);
    __syncthreads();
    if (lane == 0)
#pragma unroll
      for (int c = 0; c < NV; ++c) sh[c * 32 + wid] = v[c];
  }
  __syncthreads();
  add_warps(v, sh);
}

// Block-wide sums of NV values accumulated in the kernel's precision T:
// each warp sums in T, its sums are promoted to double and warp 0 adds the
// warps' in double (fixed order).  Keeps FP64 work, which runs at a small
// fraction of the FP32 rate, to NV values per warp.  Results valid in
// thread 0 (out); sh: >= 32*NV doubles.
template <typename T, int NV>
__device__ __forceinline__ void block_sum_lo(T (&v)[NV], double (&out)[NV], double* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if constexpr (NV > 4) {
    const T t = warp_sums(v);
    __syncthreads();
    if ((lane & 3) == 0 && (lane >> 2) < NV) sh[(lane >> 2) * 32 + wid] = (double)t;
  } else {
#pragma unroll
    for (int c = 0; c < NV; ++c)
      for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_down_sync(0xffffffffu, v[c], o);
    __syncthreads();
    if (lane == 0)
#pragma unroll
      for (int c = 0; c < NV; ++c) sh[c * 32 + wid] = (double)v[c];
  }
  __syncthreads();
  add_warps(out, sh);
}

__device__ __forceinline__ double block_sum(double v, double* sh) {
  double a[1] = {v};
  block_sum_n<1>(a, sh);
  return a[0];
}

// Fixed-order sum, by one block, of the energy partials (ne doubles) and,
// if vir, of the virial partials (nw records of 6) into out[0..6].
// sh: >= 32*7 doubles.
__device__ __forceinline__ void final_reduce(const double* __restrict__ epart, long ne,
                                             const double* __restrict__ wpart, long nw, int vir,
                                             double* __restrict__ out, double* sh) {
  double v[7] = {0, 0, 0, 0, 0, 0, 0};
  for (long k = threadIdx.x; k < ne; k += blockDim.x) v[0] += epart[k];
  if (vir)
    for (long k = threadIdx.x; k < nw; k += blockDim.x)
#pragma unroll
      for (int c = 0; c < 6; ++c) v[1 + c] += wpart[6 * k + c];
  block_sum_n<7>(v, sh);
  if (threadIdx.x == 0)
    for (int c = 0; c < 7; ++c) out[c] = v[c];
}

// Eq. (last-grid-periodic-transformed) for coarsest node mu in FP64, by
// one warp: the lanes stride over nu; e_mu = sum_nu T[(mu - nu) mod n] q_nu
// and the virial record 1/2 q_mu sum_nu V[(mu - nu) mod n] q_nu.  Partial
// sums are combined by shuffles in a fixed order.
template <typename T, bool VIR>
__device__ __forceinline__ void coarsest_node(const T* __restrict__ q, int n0, int n1, int n2,
                                              const double* __restrict__ tT,
                                              const double* __restrict__ tV, T* __restrict__ e,
                                              double* __restrict__ wpart, int mu) {
  const int lane = threadIdx.x & 31;
  const int np = n0 * n1 * n2;
  const int a = mu % n0, b = (mu / n0) % n1, c = mu / (n0 * n1);
  double v[7] = {0, 0, 0, 0, 0, 0, 0};
  for (int nu = lane; nu < np; nu += 32) {
    const int a2 = nu % n0, b2 = (nu / n0) % n1, c2 = nu / (n0 * n1);
    int da = a - a2, db = b - b2, dc = c - c2;
    if (da < 0) da += n0;
    if (db < 0) db += n1;
    if (dc < 0) dc += n2;
    const int m = da + n0 * (db + n1 * dc);
    const double qv = (double)q[nu];
    v[0] += tT[m] * qv;
    if (VIR)
#pragma unroll
      for (int k = 0; k < 6; ++k) v[1 + k] += tV[(size_t)k * np + m] * qv;
  }
#pragma unroll
  for (int k = 0; k < (VIR ? 7 : 1); ++k)
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
  if (lane == 0) {
    e[mu] = (T)v[0];
    if (VIR) {
      const double hq = 0.5 * (double)q[mu];
      for (int k = 0; k < 6; ++k) wpart[6 * (size_t)mu + k] = hq * v[1 + k];
    }
  }
}

// (1/8) sqrt(binom(6, k)), the Lorentz-Berthelot expansion coefficient
// (Sec. II.D) of channel k.
__device__ __forceinline__ double lb_coef_d(int k) {
  const double b = (k == 0 || k == 6) ? 1.0 : (k == 1 || k == 5) ? 6.0 : (k == 2 || k == 4) ? 15.0
                                                                                           : 20.0;
  return 0.125 * sqrt(b);
}

// The choice of the grid part's form (see k_thin_body): the direct kernels
// where the densest surroundings of an occupied cell exceed the thinnest
// kThinRatio times, weighted by the extreme coefficients.
constexpr double kThinRatio = 16.0;

__device__ __forceinline__ double thin_range(const int* flag, int most, int least) {
  const double hi = __longlong_as_double(*(volatile const long long*)(flag + most));
  const unsigned long long k = *(volatile const unsigned long long*)(flag + least);
  return k ? hi / __longlong_as_double((long long)~k) : 1.0;
}
__device__ __forceinline__ int thin_choice(const int* flag, bool lb) {
  const int most = *(volatile const int*)(flag + kThinMax);
  const int least = kThinMany - *(volatile const int*)(flag + kThinMin);
  double r = thin_range(flag, 4, kThinC);
  if (lb) r = r * r * r * thin_range(flag, 6, kThinW);
  return (double)most * r > kThinRatio * (double)least ? 1 : 0;
}

// Fixed-point accumulation of the anterpolation: 32-bit integers for the
// FP32 modes (sums kept below 2^30), 64-bit for FP64 (below 2^61).  Each
// contribution is rounded to 2^(e-30) (FP32) or 2^(e-61) (FP64), where 2^e
// exceeds the worst-case node sum B of fixed_exponent; B is a conservative
// bound (most atoms in a cell x cells a support box meets x max |c|), so for
// FP32 the step is ~1e-6 of a typical node sum of order 1: tens of FP32
// rounding units per contribution, far below the FP32 path's force error
// but not below FP32 rounding (the bound is tested against the FP64 oracle
// on the 65,536-atom slab).  For FP64 it is ~1e-15 of a node sum.  The
// conversions stay in the kernel's own precision: FP64 arithmetic is slow on
// this GPU.
template <typename T> struct Fixed;
template <> struct Fixed<float> {
  using I = int;
  using U = unsigned int;
  static constexpr int kBits = 30;
  __device__ static float pow2(int s) { return __int_as_float((127 + s) << 23); }
  __device__ static I to_fixed(float v) { return __float2int_rn(v); }  // v already scaled
  __device__ static float from_fixed(I v, float iscale) { return (float)v * iscale; }
};
template <> struct Fixed<double> {
  using I = long long;
  using U = unsigned long long;
  static constexpr int kBits = 61;
  __device__ static double pow2(int s) { return __longlong_as_double((long long)(1023 + s) << 52); }
  __device__ static I to_fixed(double v) { return __double2ll_rn(v); }
  __device__ static double from_fixed(I v, double iscale) { return (double)v * iscale; }
};

// Scale 2^s with s chosen so that no node sum can exceed 2^kBits in
// magnitude.  |Phi| <= 1, so a node receives at most |c| per atom within 2h
// of it (per axis; with periodic images), and those atoms lie in at most
// `span` cells (cells meeting a box of width 4h), each holding at most
// flag[3] atoms: bound = flag[3] * span * max|c|.
// Lorentz-Berthelot channel m (lbm >= 0): the coefficient is
// xi_m = lbc sigma^m sqrt(2 eps), bounded by lbc sigma_max^m (flag[4..5])
// times the largest sqrt(2 eps) (flag[6..7]).
template <typename T>
__device__ __forceinline__ int fixed_exponent(const int* __restrict__ flag, double span,
                                              int lbm = -1, double lbc = 0.0) {
  double cmax = *reinterpret_cast<const double*>(flag + 4);
  if (lbm >= 0) {
    double sm = 1.0;
    for (int k = 0; k < lbm; ++k) sm *= cmax;
    cmax = lbc * sm * *reinterpret_cast<const double*>(flag + 6);
  }
  const float bound = (float)((double)flag[3] * span * cmax * (1.0 + 1e-6));
  if (!(bound > 0.f)) return 0;
  int e;
  frexpf(bound, &e);  // bound < 2^e
  return min(max(Fixed<T>::kBits - e, -120), 120);
}

// Launch with the programmatic-stream-serialization attribute (see
// pdl_begin); same semantics as kernel<<<grid, block, smem, st>>>(args...).
template <typename... KArgs, typename... Args>
inline void launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                       cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

}  // namespace mls6

// Spatial binning of the atoms (the linked-cell structure of Sec. III.D):
// wrap positions into the box, histogram them over cells of width >= a/2,
// exclusive scan of the counts, scatter into cell order, and order each
// cell (FP32 by x, FP64 by input index) so that every later sum runs in a
// reproducible order.
#include <algorithm>
#include <climits>

#include "mls6_device.cuh"

namespace mls6 {


template <typename T> struct BinArgs {
  Box3<T> box;
  T inv_w[3];
  int nc[3];
};

// Also keeps, for the fixed-point anterpolation, the largest |c| in
// flag[4..5] (a double; one atomic maximum per block on its bits, which
// order like the value for non-negative doubles), the least nonzero |c| in
// flag[kThinC..] (for k_thin), and, when tsum is given
// (at most kScanDirect tiles), adds the block's atoms per scan tile of
// kScanTile cells to tsum (a shared-memory histogram first, then one
// integer atomic per touched tile).  count, flag and tsum start at zero (one
// memset of the region they share, per evaluation).  cell_of keeps each
// atom's cell and its place among the cell's atoms (the count it met), so
// that the scatter needs no atomics of its own.
template <typename T>
__device__ __forceinline__ void k_bin_body(const Blk bk,const T* __restrict__ pos, const T* __restrict__ cc, int stride, int N,
                      BinArgs<T> g, Vec4<T>* __restrict__ posw, int2* __restrict__ cell_of,
                      int* __restrict__ count, int* __restrict__ flag, int* __restrict__ tsum,
                      int ntiles) {
  const long z = pdl_begin();
  pos += z; cc += z;
  __shared__ T wmax[32], wmin[32];
  __shared__ int hist[kScanDirect];
  const int i = bk.x * blockDim.x + threadIdx.x;
  if (tsum)
    for (int t = threadIdx.x; t < ntiles; t += blockDim.x) hist[t] = 0;
  __syncthreads();
  T cabs = T(0);
  if (i < N) {
    const T* p = pos + (size_t)i * stride;
    T x = p[0], y = p[1], z = p[2];
    T c = cc ? cc[i] : p[3];
    if (!(isfinite(x) && isfinite(y) && isfinite(z) && isfinite(c))) {
      atomicOr(flag, 1);
      x = y = z = c = T(0);
    }
    x = wrapx(x, g.box.L[0], g.box.invL[0]);
    y = wrapx(y, g.box.L[1], g.box.invL[1]);
    z = wrapx(z, g.box.L[2], g.box.invL[2]);
    int cx = min(max((int)(x * g.inv_w[0]), 0), g.nc[0] - 1);
    int cy = min(max((int)(y * g.inv_w[1]), 0), g.nc[1] - 1);
    int cz = min(max((int)(z * g.inv_w[2]), 0), g.nc[2] - 1);
    int cell = cx + g.nc[0] * (cy + g.nc[1] * cz);
    Vec4<T> v;
    v.x = x;
    v.y = y;
    v.z = z;
    v.w = c;
    posw[i] = v;
    cell_of[i] = make_int2(cell, atomicAdd(&count[cell], 1));
    if (tsum) atomicAdd(&hist[cell / kScanTile], 1);
    cabs = fabs(c);
  }
  T cmin = cabs > T(0) ? cabs : T(INFINITY);
  warp_range(cmin, cabs);
  if ((threadIdx.x & 31) == 0) {
    wmax[threadIdx.x >> 5] = cabs;
    wmin[threadIdx.x >> 5] = cmin;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    T m = T(0), lo = T(INFINITY);
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      m = fmax(m, wmax[w]);
      lo = fmin(lo, wmin[w]);
    }
    raise_to(reinterpret_cast<unsigned long long*>(flag + 4),
             (unsigned long long)__double_as_longlong((double)m));
    if (lo <= m)  // else no atom with a coefficient
      raise_to(reinterpret_cast<unsigned long long*>(flag + kThinC),
               ~(unsigned long long)__double_as_longlong((double)lo));
  }
  if (tsum)
    for (int t = threadIdx.x; t < ntiles; t += blockDim.x)
      if (hist[t]) atomicAdd(&tsum[t], hist[t]);
}

template <typename T>
__global__ void k_bin(const T* __restrict__ pos, const T* __restrict__ cc, int stride, int N,
                      BinArgs<T> g, Vec4<T>* __restrict__ posw, int2* __restrict__ cell_of,
                      int* __restrict__ count, int* __restrict__ flag, int* __restrict__ tsum,
                      int ntiles) {
  k_bin_body<T>(Blk::self(), pos, cc, stride, N, g, posw, cell_of, count, flag, tsum, ntiles);
}

// Tile pass, for more than kScanDirect tiles: per-tile sums of the cell
// counts; the last block to finish (ticket counter, reset by that block)
// turns them into exclusive tile offsets (block-wide scan, blockDim.x tiles
// at a time with a running carry) and writes the grand total to start[n].
__device__ __forceinline__ void k_scan_tiles_body(const Blk bk,const int* __restrict__ count, long n, int* __restrict__ tsum,
                             int* __restrict__ start, int* __restrict__ flag) {
  const long z = pdl_begin();
  count += z;
  __shared__ int shm[32];
  __shared__ bool last;
  unsigned* ticket = reinterpret_cast<unsigned*>(flag + 2);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const long base = (long)bk.x * kScanTile;
  int s = 0;
  for (int t = threadIdx.x; t < kScanTile; t += blockDim.x)
    if (base + t < n) s += count[base + t];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) shm[wid] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    int tot = 0;
    for (int w = 0; w < nw; ++w) tot += shm[w];
    tsum[bk.x] = tot;
    __threadfence();
    last = atomicAdd(ticket, 1u) == bk.n - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  int carry = 0;
  for (int t0 = 0; t0 < (int)bk.n; t0 += blockDim.x) {
    const int t = t0 + threadIdx.x;
    const int v = t < (int)bk.n ? ((volatile int*)tsum)[t] : 0;
    int incl = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    __syncthreads();  // shm free (previous chunk / tile sums above)
    if (lane == 31) shm[wid] = incl;
    __syncthreads();
    int wbase = 0, total = 0;
    for (int w = 0; w < nw; ++w) {
      const int ws = shm[w];
      if (w < wid) wbase += ws;
      total += ws;
    }
    if (t < (int)bk.n) tsum[t] = carry + wbase + incl - v;
    carry += total;
  }
  if (threadIdx.x == 0) {
    start[n] = carry;
    *ticket = 0u;
  }
}

#ifndef MLS6_DEVICE_ONLY  // non-template kernel, left out where another unit includes this file
__global__ void k_scan_tiles(const int* __restrict__ count, long n, int* __restrict__ tsum,
                             int* __restrict__ start, int* __restrict__ flag) {
  k_scan_tiles_body(Blk::self(), count, n, tsum, start, flag);
}
#else
__global__ void k_scan_tiles(const int* __restrict__ count, long n, int* __restrict__ tsum,
                             int* __restrict__ start, int* __restrict__ flag);
#endif  // MLS6_DEVICE_ONLY

// Scan inside each tile (256 threads x 8 consecutive cells), write start[],
// and keep the largest cell population in flag[3] (one atomic maximum per block).  The
// tile's offset is tsum[tile] from the tile pass, or (direct: at most
// kScanDirect tiles, tsum holding the tile sums from the binning) the sum of
// the preceding tiles' sums, formed by each block; the last tile then also
// writes the grand total to start[n].
__device__ __forceinline__ void k_scan_final_body(const Blk bk,const int* __restrict__ count, long n, const int* __restrict__ tsum,
                             int* __restrict__ start, int direct, int* __restrict__ flag) {
  const long z = pdl_begin();
  tsum += z;
  count += z;
  __shared__ int wsum[32], wmx[32];
  __shared__ int toff;
  constexpr int PER = kScanTile / 256;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  long base = (long)bk.x * kScanTile + (long)threadIdx.x * PER;
  int v[PER], s = 0, mx = 0;
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    v[k] = (base + k < n) ? count[base + k] : 0;
    s += v[k];
    mx = max(mx, v[k]);
  }
  int pre = 0;  // direct: this thread's share of the preceding tiles' sums
  if (direct)
    for (int t = threadIdx.x; t < (int)bk.x; t += blockDim.x) pre += tsum[t];
  for (int o = 16; o > 0; o >>= 1) {
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    pre += __shfl_xor_sync(0xffffffffu, pre, o);
  }
  int incl = s;
  for (int o = 1; o < 32; o <<= 1) {
    int u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) wsum[wid] = incl;
  if (lane == 0) wmx[wid] = direct ? pre : 0;
  __syncthreads();
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int w = 0; w < nw; ++w) acc += wmx[w];
    toff = direct ? acc : tsum[bk.x];
  }
  if (wid == 0) {
    int x = lane < nw ? wsum[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      int u = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += u;
    }
    wsum[lane] = x;
  }
  __syncthreads();
  if (lane == 0) wmx[wid] = mx;  // wmx read above by thread 0 before this barrier
  int excl = incl - s + (wid > 0 ? wsum[wid - 1] : 0) + toff;
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    if (base + k < n) start[base + k] = excl;
    excl += v[k];
  }
  if (direct && threadIdx.x == blockDim.x - 1 && bk.x == bk.n - 1) start[n] = excl;
  __syncthreads();
  if (threadIdx.x == 0) {
    int m = 0;
    for (int w = 0; w < nw; ++w) m = max(m, wmx[w]);
    atomicMax(flag + 3, m);
  }
}

#ifndef MLS6_DEVICE_ONLY  // non-template kernel, left out where another unit includes this file
__global__ void k_scan_final(const int* __restrict__ count, long n, const int* __restrict__ tsum,
                             int* __restrict__ start, int direct, int* __restrict__ flag) {
  k_scan_final_body(Blk::self(), count, n, tsum, start, direct, flag);
}
#else
__global__ void k_scan_final(const int* __restrict__ count, long n, const int* __restrict__ tsum,
                             int* __restrict__ start, int direct, int* __restrict__ flag);
#endif  // MLS6_DEVICE_ONLY

// Input indices into cell order; the records follow them in the cell sort.
__device__ __forceinline__ void k_scatter_body(const Blk bk,const int2* __restrict__ cell_of, int N,
                          const int* __restrict__ start, int* __restrict__ sidx) {
  const long z = pdl_begin();
  cell_of += z; start += z;
  const int i = bk.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int2 c = cell_of[i];
  sidx[start[c.x] + c.y] = i;
}

#ifndef MLS6_DEVICE_ONLY  // non-template kernel, left out where another unit includes this file
__global__ void k_scatter(const int2* __restrict__ cell_of, int N, const int* __restrict__ start,
                          int* __restrict__ sidx) {
  k_scatter_body(Blk::self(), cell_of, N, start, sidx);
}
#else
__global__ void k_scatter(const int2* __restrict__ cell_of, int N, const int* __restrict__ start,
                          int* __restrict__ sidx);
#endif  // MLS6_DEVICE_ONLY

// Cell records in their final order, taken from the input-order records: FP32
// plans by x (ties by input index), so that consecutive atoms of a row of
// cells lie close together along x (the tile form of the pair sum evaluates 8
// of them against their common neighbours: 511 -> 494 candidates and 315 ->
// 298 listed ones per 8 atoms at a = 3, density 0.85); FP64 plans by input
// index.  Either way every later sum runs in an order that does not depend on
// the atomics of the binning.  Cells of up to 8 atoms (nearly all at liquid
// densities with cells of width a/2) sort 64-bit keys (the bits of x >= 0 over
// the index) in registers by an odd-even transposition network and only then
// copy the records; in larger cells every atom counts the smaller keys of its
// cell (one thread per atom, the cell's keys from L1); cells above 256 atoms
// are left in scatter order (results stay correct, only bitwise reproducibility
// is lost for them).  Threads that count are those of the block that has the
// cells, or, from kSlotAtoms atoms per cell on, of blocks of their own (a block
// of 256 cells would take thousands of atoms).  FP64 plans also get
// the positions in FP32, for the cutoff test of the pair sum's queue form.
template <typename T>
__device__ __forceinline__ unsigned long long record_key(const Vec4<T>* __restrict__ posw, int i) {
  unsigned long long k = (unsigned)i;
  if constexpr (sizeof(T) == 4) k |= (unsigned long long)__float_as_uint(posw[i].x) << 32;
  return k;
}

template <typename T>
__device__ __forceinline__ void put_record(Vec4<T>* sorted, float4* sortedf, int k, const Vec4<T>& v) {
  sorted[k] = v;
  if constexpr (sizeof(T) == 8)
    sortedf[k] = make_float4((float)v.x, (float)v.y, (float)v.z, 0.f);
}

// The atom in slot k, if its cell has more than 8: its place among the cell's.
// slots: scatter-order indices, sidx: the cell order's.
template <typename T>
__device__ __forceinline__ void rank_in_cell(const int* __restrict__ start,
                           const int2* __restrict__ cell_of, const Vec4<T>* __restrict__ posw,
                           Vec4<T>* __restrict__ sorted, const int* __restrict__ slots,
                           int* __restrict__ sidx, float4* __restrict__ sortedf, int k) {
  const int i = slots[k];
  const int c = cell_of[i].x;
  const int b = start[c], e = start[c + 1];
  if (e - b <= 8) return;
  int at = k;
  if (e - b <= 256) {
    const unsigned long long key = record_key(posw, i);
    at = b;
#pragma unroll 4
    for (int j = b; j < e; ++j) at += record_key(posw, slots[j]) < key ? 1 : 0;
  }
  sidx[at] = i;
  put_record(sorted, sortedf, at, posw[i]);
}

// big: the block also takes the atoms of its cells of more than 8.
template <typename T>
__device__ __forceinline__ void k_cellsort_body(const Blk bk,const int* __restrict__ start, long ncell,
                           const int2* __restrict__ cell_of, const Vec4<T>* __restrict__ posw,
                           Vec4<T>* __restrict__ sorted, const int* __restrict__ slots,
                           int* __restrict__ sidx, float4* __restrict__ sortedf, bool big) {
  const long z = pdl_begin();
  start += z; posw += z; cell_of += z; slots += z;
  const long first = (long)bk.x * blockDim.x, cell = first + threadIdx.x;
  const int b = cell < ncell ? start[cell] : 0, n = cell < ncell ? start[cell + 1] - b : 0;
  if (n <= 8) {
    unsigned long long key[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      key[k] = ~0ull;
      if (k < n) key[k] = record_key(posw, slots[b + k]);
    }
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int k = r & 1; k + 1 < 8; k += 2)
        if (key[k] > key[k + 1]) {
          const unsigned long long t = key[k];
          key[k] = key[k + 1];
          key[k + 1] = t;
        }
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (k < n) {
        const int i = (int)(unsigned)key[k];
        sidx[b + k] = i;
        put_record(sorted, sortedf, b + k, posw[i]);
      }
  }
  if (big && __syncthreads_or(n > 8)) {
    const int lo = start[first], hi = start[min(ncell, first + (long)blockDim.x)];
    for (int k = lo + threadIdx.x; k < hi; k += blockDim.x)
      rank_in_cell<T>(start, cell_of, posw, sorted, slots, sidx, sortedf, k);
  }
}

// Which form the grid part takes.  A transform spreads the rounding of the
// largest potentials over the whole box, where the direct kernels round each
// node's sum relative to itself: with atoms in a thin phase beside a dense one
// (a vapour, far from a droplet or a slab) their forces from transforms would
// be 5 to 9 times further off (relative to themselves; atoms near others are
// dominated by the rounding of the pair sum).  So the direct kernels run where
// the densest surroundings of an occupied cell (atoms in the 3 x 3 x 3 cells
// around it) exceed the thinnest kThinRatio times, each weighted by the
// extreme coefficients.  Surfaces of slabs reach 5 (with C6 in 0.5 .. 1.5: 8),
// single atoms of a vapour 20 to 100.  Lorentz-Berthelot: C grows like sigma^3
// sqrt(eps) of either atom.  One thread per cell, in blocks of their own beside
// the cell sort's; the anterpolation decides (k_anterp_body).
struct ThinArgs {
  int nc[3];
};

__device__ __forceinline__ void k_thin_body(const Blk bk, const int* __restrict__ start, long ncell,
                                            ThinArgs g, int* __restrict__ flag) {
  const long z0 = pdl_begin();
  start += z0;
  __shared__ int smax[32], smin[32];
  const long cell = (long)bk.x * blockDim.x + threadIdx.x;
  const bool occ = cell < ncell && start[cell + 1] > start[cell];
  int n = 0;
  if (occ) {
    int x, y, z;
    if (ncell <= 0x7fffffff) {  // 64-bit divisions are long
      const unsigned c = (unsigned)cell, q = c / (unsigned)g.nc[0];
      x = (int)(c - q * (unsigned)g.nc[0]);
      y = (int)(q % (unsigned)g.nc[1]);
      z = (int)(q / (unsigned)g.nc[1]);
    } else {
      const long q = cell / g.nc[0];
      x = (int)(cell - q * g.nc[0]);
      y = (int)(q % g.nc[1]);
      z = (int)(q / g.nc[1]);
    }
    n = atoms_around(start, g.nc, x, y, z);
  }
  const int mx = __reduce_max_sync(0xffffffffu, n);
  const int mn = __reduce_max_sync(0xffffffffu, occ ? kThinMany - n : 0);
  if ((threadIdx.x & 31) == 0) {
    smax[threadIdx.x >> 5] = mx;
    smin[threadIdx.x >> 5] = mn;
  }
  __syncthreads();
  if (threadIdx.x > 0) return;
  int hi = 0, lo = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
    hi = max(hi, smax[w]);
    lo = max(lo, smin[w]);
  }
  if (hi > 0) {
    raise_to(flag + kThinMax, hi);
    raise_to(flag + kThinMin, lo);
  }
}

// Blocks: what the choice of the grid part's form needs (if any; first, so that
// their loads run beside the sort's), cells, atoms of large cells (if any blocks
// are theirs).
template <typename T>
__global__ void k_cellsort(const int* __restrict__ start, long ncell,
                           const int2* __restrict__ cell_of, const Vec4<T>* __restrict__ posw,
                           Vec4<T>* __restrict__ sorted, const int* __restrict__ slots,
                           int* __restrict__ sidx, float4* __restrict__ sortedf, int N, int nthin,
                           int ncells, int nslots, ThinArgs g, int* __restrict__ flag) {
  const int b = (int)blockIdx.x - nthin;
  if (b < 0) {
    k_thin_body(Blk{blockIdx.x, (unsigned)nthin}, start, ncell, g, flag);
  } else if (b < ncells) {
    k_cellsort_body<T>(Blk{(unsigned)b, (unsigned)ncells}, start, ncell, cell_of, posw, sorted,
                       slots, sidx, sortedf, nslots == 0);
  } else {
    const long z = pdl_begin();
    const int k = (b - ncells) * blockDim.x + threadIdx.x;
    if (k < N)
      rank_in_cell<T>(start + z, cell_of + z, posw + z, sorted, slots + z, sidx, sortedf, k);
  }
}

static ThinArgs thin_args(const Plan* p) {
  return ThinArgs{{p->cg.nc[0], p->cg.nc[1], p->cg.nc[2]}};
}

// Atoms per cell from which the atoms of large cells get blocks of their own.
// Binning stage, 100,000 atoms in FP32, with an insertion sort per cell (one
// thread, two dependent loads per comparison) -> here: 6.8 atoms per cell
// (a = 4) 39 -> 19 us (30 without blocks of their own), 13 (a = 5) 92 -> 21, 54
// (a = 8) 911 -> 26; cells of 370 atoms, copied by one thread each, 2588 -> 26.
// Between 4 and 6 atoms per cell the two agree.
constexpr long kSlotAtoms = 6;

// Scatter-order indices: in the pair sum's output, which is written later.
static int* scatter_slots(const Plan* p) { return reinterpret_cast<int*>(p->d_floc); }

// Arguments of the binning kernel for a plan.
template <typename T> static BinArgs<T> bin_args(const Plan* p) {
  BinArgs<T> bg;
  for (int d = 0; d < 3; ++d) {
    bg.box.L[d] = (T)p->L[d];
    bg.box.invL[d] = (T)(1.0 / p->L[d]);
    bg.inv_w[d] = (T)p->cg.inv_w[d];
    bg.nc[d] = p->cg.nc[d];
  }
  return bg;
}

template <typename T>
int launch_bin(Plan* p, const T* pos, const T* cc, cudaStream_t st) {
  const int N = (int)p->N;
  const BinArgs<T> bg = bin_args<T>(p);
  const long ncell = p->cg.ncell;
  const long ntiles = cdiv(ncell, kScanTile);
  // direct: tile sums from the binning, no tile pass
  const bool direct = ntiles <= kScanDirect;
  const int nbin = (int)cdiv(N, kBlock);
  launch_pdl(k_bin<T>, nbin, kBlock, 0, st, pos, cc, cc ? 3 : 4, N, bg, (Vec4<T>*)p->d_pos_w,
             p->d_cell_of, p->d_cell_count, p->d_flag, direct ? p->d_scan : (int*)nullptr,
             (int)ntiles);
  if (!direct)
    launch_pdl(k_scan_tiles, ntiles, kBlock, 0, st, (const int*)p->d_cell_count, ncell, p->d_scan,
               p->d_cell_start, p->d_flag);
  launch_pdl(k_scan_final, ntiles, kBlock, 0, st, (const int*)p->d_cell_count, ncell, (const int*)p->d_scan,
             p->d_cell_start, direct ? 1 : 0, p->d_flag);
  int* slots = scatter_slots(p);
  launch_pdl(k_scatter, cdiv(N, kBlock), kBlock, 0, st, (const int2*)p->d_cell_of, N,
             (const int*)p->d_cell_start, slots);
  const int ncells = (int)cdiv(ncell, kBlock);
  const int nslots = N >= kSlotAtoms * ncell ? (int)cdiv(N, kBlock) : 0;
  const int nthin = p->spectral ? ncells : 0;
  launch_pdl(k_cellsort<T>, nthin + ncells + nslots, kBlock, 0, st, (const int*)p->d_cell_start,
             ncell, (const int2*)p->d_cell_of, (const Vec4<T>*)p->d_pos_w,
             (Vec4<T>*)p->d_sorted, (const int*)slots, p->d_sorted_idx, (float4*)p->d_sorted_f, N,
             nthin, ncells, nslots, thin_args(p), p->d_flag);
  return direct ? 4 : 5;
}

#ifndef MLS6_DEVICE_ONLY  // host code, left out where another unit includes this file
template int launch_bin<float>(Plan*, const float*, const float*, cudaStream_t);
template int launch_bin<double>(Plan*, const double*, const double*, cudaStream_t);

#endif  // MLS6_DEVICE_ONLY
}  // namespace mls6

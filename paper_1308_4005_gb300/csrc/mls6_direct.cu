// The direct grid part of one plan in one launch: restriction, the level
// stencils, the coarsest level and prolongation (mls6_grid.cu's kernel bodies),
// for evaluations with thin phases of a plan that has the transforms
// (thin_choice, mls6_device.cuh).
//
// A work queue of (stage, block) items, numbered stage by stage.  A block takes
// the next number with one atomic ticket and, before it runs the item, waits
// until the stage before has counted all its blocks done.  Every item that a
// block waits for has a smaller number and so was taken by a block that is
// running: the queue cannot deadlock, whatever the number of resident blocks.
// The waits are bounded all the same (MLS6_ERR_TIMEOUT).
//
// This unit compiles the kernel bodies without the __restrict__ qualifiers, so
// that no load of data written earlier in the same launch (by other blocks) can
// go through the non-coherent read-only path; producers publish with a fence
// before they count, and the polling thread fences after it sees the count.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <vector>

#define __restrict__
#define MLS6_DEVICE_ONLY
#include "mls6_bin.cu"
#include "mls6_grid.cu"
#undef MLS6_DEVICE_ONLY
#undef __restrict__

namespace mls6 {

// One launch, because it is part of every evaluation and mostly finds that it
// has nothing to do: with the choice it costs 1 of 53 us at 3,001 atoms, 2 of 87
// at 65,536, 12 of 765 at 1,048,576, where its blocks wait for room beside the
// pair sum's (on a stream of its own beside the transforms, or behind the pair
// sum: the same or more).  With a vapour, whole
// evaluations, with the separate launches (and the pair sums of that time) ->
// here: 3,001-atom slab 88 -> 99 us (the transforms' launches that return at
// once), 65,536 atoms 162 -> 140, FP64 20,000 788 -> 427, 1,000,000 atoms 1232 ->
// 1096.  Bound like those by latency on small grids and
// by the stencil's FP32 pipe on large ones, so 64 registers, as its kernel has
// (128: 65,536 atoms 172).  The level stencils' tensor-core forms stay out: they
// round coarser.
enum GKind : int { G_FROM_FIXED, G_RESTRICT, G_STENCIL, G_TOP, G_PROLONG };

struct GStage {
  int kind;
  unsigned nb;
  long long first;            // its first item
  const void *a, *b;          // sums | q^k | e^k, e^{k+1,tot}
  void* out;
  int f[3], c[3];             // nodes of the finer and the coarser grid
  int lbm;                    // Lorentz-Berthelot channel, or -1
  double lbc;
};

template <typename T> struct DirectArgs {
  StencilArgs<T> A;
  const GStage* st;
  int S;
  long long total, limit;
  PQueue* q;
  unsigned* done;
  int* flag;
  double span;
  double* wsten;
  long nodes;                 // of the levels below the coarsest (global-memory stencil)
  int global;
};

// G: thread groups per stencil tile, the plan's (a plan with one takes two).
template <typename T, int NP, bool VIR, int G>
__global__ void __launch_bounds__(kStencilThreads * G, sizeof(T) == 4 ? 8 / G : 1)
    k_direct(const __grid_constant__ DirectArgs<T> X) {
  __shared__ int s_stage;
  __shared__ unsigned s_block;
  pdl_begin();
  if (*(volatile const int*)(X.flag + kThin) == 0) return;
  for (;;) {
    if (threadIdx.x == 0) {
      const long long t = (long long)atomicAdd(&X.q->ticket, 1ull);
      int lo = -1;
      if (t < X.total) {
        lo = 0;
        for (int hi = X.S; hi - lo > 1;) {
          const int mid = (lo + hi) >> 1;
          if (X.st[mid].first <= t) lo = mid;
          else hi = mid;
        }
        s_block = (unsigned)(t - X.st[lo].first);
        for (long long it = 0; lo > 0; ++it) {
          if (ld_acquire(X.done + lo - 1) >= X.st[lo - 1].nb) break;
          if (it >= X.limit || *(volatile int*)&X.q->error) {  // reported as MLS6_ERR_TIMEOUT
            atomicOr(&X.q->error, 1);
            atomicOr(X.flag, 2);
            lo = -1;
            break;
          }
          __nanosleep(20);
        }
      }
      __threadfence();
      s_stage = lo;
    }
    __syncthreads();
    const int s = s_stage;
    if (s < 0) return;
    const GStage& d = X.st[s];
    const Blk bk{s_block, d.nb};
    switch (d.kind) {
      case G_FROM_FIXED:
        k_from_fixed_body<T>(bk, (const typename Fixed<T>::U*)d.a, (long)d.f[0] * d.f[1] * d.f[2],
                             X.flag, X.span, (T*)d.out, d.lbm, d.lbc);
        break;
      case G_RESTRICT:
        k_restrict_body<T, NP>(bk, (const T*)d.a, d.f[0], d.f[1], d.f[2], (T*)d.out, d.c[0],
                               d.c[1], d.c[2]);
        break;
      case G_STENCIL:
        if (X.global)
          k_stencil_global_body<T, VIR>(bk, X.A, X.wsten, X.nodes);
        else
          k_stencil_body<T, VIR, G>(bk, X.A, X.wsten);
        break;
      case G_TOP: {
        const int mu = (int)bk.x * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5);
        if (mu < X.A.nt[0] * X.A.nt[1] * X.A.nt[2])
          coarsest_node<T, VIR>(X.A.qt, X.A.nt[0], X.A.nt[1], X.A.nt[2], X.A.tT, X.A.tV, X.A.et,
                                X.A.wtop, mu);
        break;
      }
      default:
        k_prolong_body<T, NP>(bk, (const T*)d.a, d.f[0], d.f[1], d.f[2], (const T*)d.b, d.c[0],
                              d.c[1], d.c[2], (T*)d.out);
        break;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      atomicAdd(X.done + s, 1u);
    }
  }
}

// The stencil's geometry: 8^3 tiles, or nodes where the tile and the taps do
// not fit in shared memory (the plan's own may be that of the tensor cores).
struct DirectGeometry {
  bool global;
  size_t smem;
  long blocks, nodes;
  int tiles[kMaxLevels + 1][3];
  long off[kMaxLevels + 1];
};

static DirectGeometry direct_geometry(const Plan* p, int threads) {
  DirectGeometry G;
  const int S = kStencilTile + 2 * p->P;
  int Sx, Sp;
  stencil_pitches(S, Sx, Sp);
  G.smem = align16(p->elem() * S * Sp) + 4 * p->elem() * p->ntaps + sizeof(int4) * p->nrows;
  G.global = G.smem > kStencilSmemMax;
  if (G.global) G.smem = 0;
  G.blocks = G.nodes = 0;
  for (int k = 1; k < p->levels; ++k) {
    long nt = 1;
    for (int d = 0; d < 3; ++d) {
      G.tiles[k][d] = (int)cdiv(p->lv[k].n[d], kStencilTile);
      nt *= G.tiles[k][d];
    }
    G.off[k] = G.blocks;
    G.blocks += nt;
    G.nodes += p->lv[k].np;
  }
  if (G.global) G.blocks = cdiv(G.nodes, threads);
  return G;
}

static int direct_threads(int i) { return kStencilThreads * (i ? 4 : 2); }

long direct_records(const Plan* p) { return direct_geometry(p, direct_threads(0)).blocks; }

// Queue and counters, for a Lorentz-Berthelot evaluation (seven channels).
size_t direct_queue_bytes(const Plan* p) {
  return sizeof(PQueue) + sizeof(unsigned) * 7 * (2 * p->levels + 1);
}

template <typename T> using DirectKernel = void (*)(DirectArgs<T>);
template <typename T, int G> static DirectKernel<T> direct_kernel(const Plan* p, bool vir) {
  if (p->order == 5) return vir ? k_direct<T, 6, true, G> : k_direct<T, 6, false, G>;
  return vir ? k_direct<T, 4, true, G> : k_direct<T, 4, false, G>;
}
template <typename T> static DirectKernel<T> direct_kernel(const Plan* p, int i, bool vir) {
  return i ? direct_kernel<T, 4>(p, vir) : direct_kernel<T, 2>(p, vir);
}

// Stage list for blocks of direct_threads(i).
template <typename T> static int prepare_direct_list(Plan* p, bool lb, int i) {
  const int nt = direct_threads(i);
  const DirectGeometry G = direct_geometry(p, nt);
  const int l = p->levels;
  const Level& L1 = p->lv[1];
  Plan::DirectGrid& g = p->direct[lb][i];
  std::vector<GStage> st;
  long long first = 0;
  auto add = [&](int kind, long nb, const void* a, const void* b, void* out, const Level& f,
                 const Level& c) -> GStage& {
    GStage s = {};
    s.kind = kind;
    s.nb = (unsigned)nb;
    s.first = first;
    s.a = a;
    s.b = b;
    s.out = out;
    for (int d = 0; d < 3; ++d) {
      s.f[d] = f.n[d];
      s.c[d] = c.n[d];
    }
    s.lbm = -1;
    first += nb;
    st.push_back(s);
    return st.back();
  };
  for (int m = 0; m < (lb ? 7 : 1); ++m) {
    const T* sums = lb ? (const T*)p->d_lbq + (size_t)m * L1.np : (const T*)p->d_q1fx;
    GStage& s = add(G_FROM_FIXED, cdiv(L1.np, nt), sums, nullptr, p->d_q[1], L1, L1);
    if (lb) {
      s.lbm = m;
      s.lbc = lb_coef(m);
    }
    for (int k = 1; k < l; ++k)
      add(G_RESTRICT, cdiv(p->lv[k + 1].np, nt), p->d_q[k], nullptr, p->d_q[k + 1], p->lv[k],
          p->lv[k + 1]);
    const long top = cdiv(p->lv[l].np, nt / 32);
    add(G_STENCIL, G.blocks + (G.global ? 0 : top), nullptr, nullptr, nullptr, L1, L1);
    if (G.global) add(G_TOP, top, nullptr, nullptr, nullptr, L1, L1);
    for (int k = l - 1; k >= 1; --k)
      add(G_PROLONG, cdiv(p->lv[k].np, nt), p->d_e[k], p->d_et[k + 1],
          lb && k == 1 ? (void*)((T*)p->d_lbpot + (size_t)m * L1.np) : p->d_et[k], p->lv[k],
          p->lv[k + 1]);
  }
  // blocks: up to two per SM, at most what a stage has (four per SM: 1,000,000
  // atoms with a vapour 1127 us against 1096; one: 1650, 65,536 atoms 152 against 140)
  unsigned most = 1;
  for (const GStage& s : st) most = std::max(most, s.nb);
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return MLS6_ERR_CUDA;
  for (int v = 0; v < 2; ++v) {
    const DirectKernel<T> kern = direct_kernel<T>(p, i, v);
    int per_sm = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kStencilSmemMax) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nt, G.smem) != cudaSuccess ||
        per_sm < 1)
      return MLS6_ERR_CUDA;
    g.blocks[v] = (int)std::min<long>((long)most, (long)std::min(per_sm, 2) * sms);
  }
  void* d_st = nullptr;
  const size_t bytes = sizeof(GStage) * st.size();
  if (cudaMalloc(&d_st, bytes) != cudaSuccess) {
    cudaGetLastError();
    return MLS6_ERR_NOMEM;
  }
  if (cudaMemcpy(d_st, st.data(), bytes, cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaFree(d_st);
    return MLS6_ERR_CUDA;
  }
  g.d_stages = d_st;
  g.stages = (int)st.size();
  g.items = first;
  return MLS6_OK;
}

// (the list of four groups last: it is there when both are)
template <typename T> int prepare_direct(Plan* p, bool lb) {
  for (int i = 0; i < 2; ++i)
    if (!p->direct[lb][i].d_stages) {
      const int rc = prepare_direct_list<T>(p, lb, i);
      if (rc) return rc;
    }
  return MLS6_OK;
}
template int prepare_direct<float>(Plan*, bool);
template int prepare_direct<double>(Plan*, bool);

template <typename T> int launch_direct(Plan* p, bool vir, bool lb, cudaStream_t st) {
  const int i = p->stencil_groups > 2 ? 1 : 0, nt = direct_threads(i);
  const DirectGeometry G = direct_geometry(p, nt);
  const Plan::DirectGrid& g = p->direct[lb][i];
  DirectArgs<T> X;
  X.A = stencil_args<T>(p);
  if (!G.global)
    for (int k = 1; k < p->levels; ++k) {
      for (int d = 0; d < 3; ++d) X.A.lv[k - 1].tiles[d] = G.tiles[k][d];
      X.A.lv[k - 1].tile_off = G.off[k];
    }
  X.A.sblocks = G.blocks;
  X.st = reinterpret_cast<const GStage*>(g.d_stages);
  X.S = g.stages;
  X.total = g.items;
  X.limit = 1LL << 24;
  X.q = reinterpret_cast<PQueue*>(p->d_direct_queue);
  X.done = reinterpret_cast<unsigned*>(p->d_direct_queue + sizeof(PQueue));
  X.flag = p->d_flag;
  X.span = support_span(p);
  X.wsten = p->d_wpart + 6 * p->wpart_stencil;
  X.nodes = G.nodes;
  X.global = G.global ? 1 : 0;
  launch_pdl(direct_kernel<T>(p, i, vir), g.blocks[vir], nt, G.smem, st, X);
  return 1;
}
template int launch_direct<float>(Plan*, bool, bool, cudaStream_t);
template int launch_direct<double>(Plan*, bool, bool, cudaStream_t);

}  // namespace mls6
